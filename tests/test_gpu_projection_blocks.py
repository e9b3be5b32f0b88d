"""The set-up, projection and residual kernels where their blocks end, and their dispatch on dt.

Face coefficients, correction and adjoint faces: bit for bit the oracle's (the same separately rounded
operations in the same order).  Residual norms, means and live cells: sums of n terms in another
order, each with a rounding of 2^-53 of the running sum and added in trees of blocks, so n 2^-53 (3e-12 at
the largest grid here) bounds the relative difference with room."""
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


@pytest.mark.parametrize("solid", ["none", "ellipsoid"])
@pytest.mark.parametrize("shape", [(300, 5, 20), (256, 3, 40), (33, 17, 8), (31, 1, 17), (2, 40, 3), (512, 2, 1),
                                   (64, 48, 33)])
def test_face_coeffs_blocks_bit_exact(mgp, shape, solid):
    for interface in ("random", "wave"):
        case = synth.small_case(*shape, seed=71, solid=solid, interface=interface, fields=False)
        sm = None if case.solid is None else dev(case.solid, torch.uint8)
        beta = mgp.face_coeffs(dev(case.phi), case.h, sm, rho_air=case.lam)
        for a, b in zip(faces_host(beta), O.face_coeffs(case.phi, case.solid, case.lam)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("dt", [1.0, 0.25, 0.3])
@pytest.mark.parametrize("shape", [(48, 16, 24), (16, 16, 16)])
def test_correction_and_adjoint_faces_bit_exact_for_dt(mgp, shape, dt):
    case = synth.small_case(*shape, seed=72, solid="ellipsoid")
    beta_o = O.face_coeffs(case.phi, case.solid, case.lam)
    ctx = mgp.Context(faces_dev(beta_o), case.h, coarse_max_cells=2048)
    p = np.random.default_rng(6).standard_normal(case.shape)
    for a, b in zip(faces_host(ctx.correct(faces_dev(case.u_star), dev(p), dt=dt)),
                    O.correct(beta_o, p, case.u_star, case.h, dt)):
        assert np.array_equal(a, b)
    assert np.array_equal(host(ctx.divergence(faces_dev(case.u_star), dt=dt)),
                          O.divergence(beta_o, case.u_star, case.h, dt))
    q = torch.zeros(case.shape, dtype=torch.float64, device="cuda")
    gu, gb, _ = ctx.project_adjoint(faces_dev(case.w), dev(p), dt=dt, tol=1e-8, q=q)
    gq, gp = O.gradient(beta_o, host(q), case.h), O.gradient(beta_o, p, case.h)
    for b, x, g, a, ug, bg in zip(beta_o, case.w, gq, gp, faces_host(gu), faces_host(gb)):
        assert np.array_equal(ug, np.where(b > 0, x - g, x))
        assert np.array_equal(bg, np.where(b > 0, dt * a * (g - x), 0.0))


@pytest.mark.parametrize("krylov,prec", [(0, "fp64"), (0, "mixed"), (1, "fp64"), (1, "mixed")])
@pytest.mark.parametrize("shape", [(64, 32, 16), (36, 20, 28), (5, 7, 9), (8, 8, 72), (264, 16, 16), (1, 3, 40)])
def test_residual_of_the_first_iterate(mgp, shape, krylov, prec):
    """A solve of no cycle reports the residual of its guess: a random one, one with a single nonzero
    cell, and zero."""
    case = synth.small_case(*shape, seed=73, solid="none", interface="random", fields=False)
    beta_o = O.face_coeffs(case.phi, None, case.lam)
    ctx = mgp.Context(faces_dev(beta_o), case.h, prec=prec, krylov=krylov, max_cycles=0, coarse_max_cells=2048)
    b = O.remove_mean(case.rhs, *O.components(beta_o))
    rng = np.random.default_rng(8)
    spike = np.zeros(case.shape)
    spike[-1, -1, -1] = 0.7
    for p in (rng.standard_normal(case.shape), spike, np.zeros(case.shape)):
        g, st = ctx.solve(dev(case.rhs), dev(p), tol=1e-300, allow_not_converged=True)
        n = case.ncell * 2.0 ** -53 + 1e-13
        r = np.linalg.norm(O.residual(beta_o, b, p, case.h))
        assert st.rhs_norm == pytest.approx(np.linalg.norm(b), rel=n)
        assert st.rel_resid == pytest.approx(r / np.linalg.norm(b), rel=n)
        assert np.abs(host(g) - (p - p.mean())).max() <= n * max(1.0, np.abs(p).max())


def _stretched(shape, seed, frac):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    w = [rng.uniform(0.5, 1.5, m) / m for m in shape]
    f = None
    if frac:  # open, closed and partly covered faces
        f = [np.where(rng.random((nz, ny, nx)) < 0.5, 1.0, np.maximum(rng.uniform(-0.3, 1.0, (nz, ny, nx)), 0.0))
             for _ in range(3)]
    return w, f


@pytest.mark.parametrize("frac", [False, True])
@pytest.mark.parametrize("shape", [(128, 2, 16), (129, 3, 17), (31, 5, 33), (1, 40, 15), (200, 1, 1), (2, 130, 31)])
def test_stretched_metrics_blocks_bit_exact(mgp, shape, frac):
    w, f = _stretched(shape, 74, frac)
    for interface in ("random", "wave"):
        case = synth.small_case(*shape, seed=75, solid="none", interface=interface, fields=False)
        beta = O.face_coeffs(case.phi, None, case.lam)
        bo, ao = mgp.stretched_metrics(*[dev(x) for x in w], faces_dev(beta), None if f is None else faces_dev(f))
        bi, area = O.stretched_metrics(*w, beta, f)
        for a, b in zip(faces_host(bo) + faces_host(ao), bi + area):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("shape", [(264, 16, 16), (36, 20, 28), (64, 48, 24), (32, 16, 72)])
def test_divergence_with_areas_blocks_bit_exact(mgp, shape, body):
    """Also where a closed face's velocities are not finite: such a face carries no flux."""
    case = synth.small_case(*shape, seed=76, solid="none", interface="wave")
    (hx, hy, hz), f = _stretched(shape, 77, True)
    bi, area = O.stretched_metrics(hx, hy, hz, O.face_coeffs(case.phi, None, case.lam), f)
    v = None
    if body:
        rng = np.random.default_rng(9)
        v = [rng.standard_normal(case.shape) for _ in range(3)]
    ctx = mgp.Context(faces_dev(bi), 1.0, krylov=1, coarse_max_cells=2048)
    ctx.set_face_areas(faces_dev(area))
    if body:
        ctx.set_body_velocity(faces_dev(v))
    want = O.divergence_area(area, case.u_star, 1.0, 0.3, v)
    u = [np.where(a > 0, x, np.inf) for a, x in zip(area, case.u_star)]
    assert np.array_equal(host(ctx.divergence(faces_dev(u), dt=0.3)), want)
