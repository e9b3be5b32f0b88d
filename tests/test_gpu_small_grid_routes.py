"""Kernels that a small grid takes cell by cell and a large one in blocks that walk up z: each side of every line,
with rows and runs that do not fill the blocks.  Bit for bit the oracle's (the same separately rounded operations in
the same order)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1410_2240_gb300 import synth

from _gpu_util import dev, faces_dev, faces_host, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mgp():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_2240_gb300 import mgproj
    return mgproj


def _areas(shape, seed):
    """Open, closed and partly covered faces."""
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    return [np.where(rng.random((nz, ny, nx)) < 0.5, 1.0, np.maximum(rng.uniform(-0.3, 1.0, (nz, ny, nx)), 0.0))
            for _ in range(3)]


@pytest.mark.parametrize("frac", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 1), (84, 84, 85), (85, 84, 84), (85, 85, 85), (300, 48, 49), (129, 171, 32),
                                   (31, 685, 33), (2, 700, 501), (700, 1001, 1), (1, 3, 70001), (1, 2, 350001),
                                   (107, 107, 105), (129, 283, 33), (1, 700, 1716)])
def test_stretched_metrics_bit_exact_on_both_routes(mgp, shape, frac):
    rng = np.random.default_rng(81)
    w = [rng.uniform(0.5, 1.5, m) / m for m in shape]
    f = _areas(shape, 82) if frac else None
    for interface in ("random", "wave"):
        case = synth.small_case(*shape, seed=83, solid="none", interface=interface, fields=False)
        beta = O.face_coeffs(case.phi, None, case.lam)
        bo, ao = mgp.stretched_metrics(*[dev(x) for x in w], faces_dev(beta), None if f is None else faces_dev(f))
        bi, area = O.stretched_metrics(*w, beta, f)
        for a, b in zip(faces_host(bo) + faces_host(ao), bi + area):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("areas,body", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("shape", [(8, 8, 8), (16, 128, 64), (32, 64, 72), (56, 56, 48), (144, 48, 40), (264, 32, 32),
                                   (160, 160, 192), (192, 160, 192)])
def test_divergence_bit_exact_on_every_route(mgp, shape, areas, body):
    case = synth.small_case(*shape, seed=84, solid="none", interface="wave", fields=False)
    rng = np.random.default_rng(85)
    field = lambda: [rng.standard_normal(case.shape) for _ in range(3)]
    f = _areas(shape, 86) if areas else [np.ones(case.shape)] * 3
    _, area = O.stretched_metrics(*[np.ones(n) for n in shape], O.face_coeffs(case.phi, None, case.lam), f)
    u, v = field(), (field() if body else None)
    ctx = mgp.Context(faces_dev(O.face_coeffs(case.phi, None, case.lam)), 1.0, coarse_max_cells=2048)
    if areas:
        ctx.set_face_areas(faces_dev(area))
    if body:
        ctx.set_body_velocity(faces_dev(v))
    for dt in (1.0, 0.3):
        assert np.array_equal(host(ctx.divergence(faces_dev(u), dt=dt)), O.divergence_area(area, u, 1.0, dt, v))


@pytest.mark.parametrize("inv_re,convection", [(0.37, True), (0.37, False), (0.0, True)])
@pytest.mark.parametrize("shape", [(1, 1, 1), (32, 33, 64), (64, 32, 35), (19, 61, 64), (20, 61, 64), (2, 190, 191),
                                   (300, 20, 13), (308, 20, 13), (96, 31, 25), (144, 144, 145), (145, 144, 144),
                                   (140, 150, 144)])
def test_momentum_bit_exact_on_every_route(mgp, shape, inv_re, convection):
    case = synth.small_case(*shape, seed=87, solid="none", interface="random", fields=False)
    rng = np.random.default_rng(88)
    u = [rng.standard_normal(case.shape) for _ in range(3)]
    beta = O.face_coeffs(case.phi, None, case.lam)
    for h in (case.h, 0.25):
        want = O.momentum_rhs(case.phi, beta, u, h, g=1.3, inv_re=inv_re, mu_air=1.8e-2, convect=convection)
        f = mgp.forces(g=1.3, inv_re=inv_re, mu_air=1.8e-2, convection=convection)
        got = mgp.momentum_rhs(dev(case.phi), faces_dev(beta), faces_dev(u), h, f)
        for a, b in zip(faces_host(got), want):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("shape", [(257, 9, 11), (300, 48, 49), (449, 5, 17), (512, 3, 9), (513, 7, 10), (705, 4, 8)])
def test_rows_of_several_blocks_bit_exact(mgp, shape):
    """Rows longer than a block are cut into equal parts of whole warps: face coefficients, their adjoint, and
    the momentum terms over the cuts."""
    case = synth.small_case(*shape, seed=89, solid="ellipsoid", interface="random", fields=False)
    rng = np.random.default_rng(90)
    field = lambda: [rng.standard_normal(case.shape) for _ in range(3)]
    for solid in (None, case.solid):
        beta = O.face_coeffs(case.phi, solid, case.lam)
        got = mgp.face_coeffs(dev(case.phi), case.h, None if solid is None else dev(solid, torch.uint8), rho_air=case.lam)
        for a, b in zip(faces_host(got), beta):
            assert np.array_equal(a, b)
        gb, u = field(), field()
        g = mgp.phi_grad(faces_dev(beta), faces_dev(gb), case.h, rho_air=case.lam)
        assert np.array_equal(host(g), O.phi_grad(beta, gb, case.lam))
        want = O.momentum_rhs(case.phi, beta, u, case.h, g=1.3, inv_re=0.37, mu_air=1.8e-2, convect=True)
        f = mgp.forces(g=1.3, inv_re=0.37, mu_air=1.8e-2, convection=True)
        for a, b in zip(faces_host(mgp.momentum_rhs(dev(case.phi), faces_dev(beta), faces_dev(u), case.h, f)), want):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("h", [0.25, 0.3])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_fused_sweeps_with_any_spacing_identical_to_passes(mgp, prec, h):
    """h^2 b is an exponent shift or a multiplication, chosen by h: the fused sweep's choice against the passes'."""
    case = synth.small_case(72, 40, 48, seed=91, solid="ellipsoid", fields=False)
    beta = mgp.face_coeffs(dev(case.phi), h, dev(case.solid, torch.uint8), rho_air=case.lam)
    rhs = dev(np.random.default_rng(92).standard_normal(case.shape))
    out = []
    for sm in (1, 2):
        ctx = mgp.Context(beta, h, prec=prec, smoother=sm, coarse_max_cells=2048)
        p = torch.zeros_like(rhs)
        for _ in range(2):
            ctx.vcycle(rhs, p)
        out.append(p)
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(5, 7, 9), (64, 32, 32), (64, 32, 40)])
def test_mean_of_p_removed_on_either_route(mgp, shape, prec):
    """A solve of no cycle returns its guess without its mean over the live cells, summed in the residual's pass or in one
    of its own: the sum of n terms is off by at most n 2^-53 of the largest of them."""
    case = synth.small_case(*shape, seed=93, solid="none" if shape[0] == 5 else "ellipsoid", fields=False)
    solid = case.solid
    beta = O.face_coeffs(case.phi, solid, case.lam)
    live = np.ones(case.shape, bool) if solid is None else solid == 0
    p = np.random.default_rng(94).standard_normal(case.shape) + 3.0
    ctx = mgp.Context(faces_dev(beta), case.h, prec=prec, max_cycles=0, coarse_max_cells=2048)
    rhs = np.where(live, np.random.default_rng(95).standard_normal(case.shape), 0.0)
    got, _ = ctx.solve(dev(rhs), dev(p), tol=1e-300, allow_not_converged=True)
    want = np.where(live, p - p[live].mean(), 0.0)
    assert np.abs(host(got) - want).max() <= p.size * 2.0 ** -53 * np.abs(p).max() + 1e-13
