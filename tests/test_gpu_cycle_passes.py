"""The passes of a V-cycle that depend on its smoothing counts: the prolongation corrects the red
cells alone where a black pass follows (nu2 >= 1), all cells otherwise; a cycle that continues
the one before it leaves its first red pass out (nu1, nu2 >= 1).

Bounds: a V-cycle against the oracle's with the same counts to 1e-12 (FP64) and 3e-6 of max|p|
(FP32), the bounds of the other cycle tests.  Cycles run by a solve against the same number of
single cycles: the kernels and their order are the same, so the iterates agree up to the mean
that the solve removes at its end (one subtraction, taken here in another order of summation):
1e-13 of max|p|.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1410_2240_gb300 import synth

from _gpu_util import case_rhs, dev, host, rel

pytestmark = pytest.mark.gpu

# cells along x: a multiple of 8, of 4 alone and of 2 alone; two to four levels; small coarsest grids
# (their oracle inverse is a dense eigen-decomposition)
SHAPES = [(48, 16, 24), (36, 16, 16), (20, 16, 24), (10, 8, 8), (16, 8, 8)]


@pytest.fixture(scope="module")
def mgp():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_2240_gb300 import mgproj
    return mgproj


def _setup(mgp, shape, **kw):
    case = synth.small_case(*shape, solid="ellipsoid", seed=51)
    beta_o = O.face_coeffs(case.phi, case.solid, case.lam)
    b = O.remove_mean(case_rhs(case, beta_o), *O.components(beta_o))
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    return case, beta_o, b, mgp.Context(beta, case.h, coarse_max_cells=2048, **kw)


@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 2), (2, 0)])
@pytest.mark.parametrize("shape", SHAPES)
def test_cycle_with_smoothing_counts_matches_oracle(mgp, shape, nu):
    for prec in ("fp64", "mixed"):
        case, beta_o, b, ctx = _setup(mgp, shape, prec=prec, nu1=nu[0], nu2=nu[1])
        mg = O.MG(beta_o, case.h, nu1=nu[0], nu2=nu[1])
        p = np.zeros(b.shape)
        for it in range(2):
            pd = dev(p)
            p = mg.vcycle(b, p)
            ctx.vcycle(dev(b), pd)
            if prec == "fp64":
                assert rel(host(pd), p) <= 1e-12, it
            else:
                assert np.abs(host(pd) - p).max() <= 3e-6 * np.abs(p).max(), it


@pytest.mark.parametrize("shape", SHAPES)
def test_continued_cycles_are_the_single_ones(mgp, shape):
    case, beta_o, b, ctx = _setup(mgp, shape, max_cycles=3)
    p, st = ctx.solve(dev(b), tol=1e-30, allow_not_converged=True)
    q = dev(np.zeros(b.shape))
    for _ in range(3):
        ctx.vcycle(dev(b), q)
    lab, nc = O.components(beta_o)
    q = O.remove_mean(host(q), lab, nc)
    assert st.cycles == 3
    assert np.abs(host(p) - q).max() <= 1e-13 * np.abs(q).max()


# first tail level (half the grid): planes that do and do not deal out evenly over 16 CTAs, fewer planes
# than CTAs, more cells per CTA than threads, the largest tail (8192 cells) and one cell more per axis,
# a coarsest grid of an odd size, one above the size the tail solves
TAIL_SHAPES = [(32, 32, 40), (16, 16, 144), (64, 64, 16), (48, 80, 24), (32, 32, 64), (36, 32, 64), (20, 24, 28),
               (44, 44, 44)]


@pytest.mark.parametrize("nu", [(2, 2), (0, 1), (1, 0)])
@pytest.mark.parametrize("shape", TAIL_SHAPES)
def test_tail_slabs_identical_to_launches(mgp, shape, nu):
    """The tail's cluster, whichever way the planes fall on its CTAs, gives the V-cycles of a launch
    per pass bit for bit (the same operations in the same order)."""
    case = synth.small_case(*shape, solid="ellipsoid", seed=52)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = dev(case.rhs)
    for prec in ("fp64", "mixed"):
        out = []
        for tail in (0, 1):
            ctx = mgp.Context(beta, case.h, prec=prec, coarse_tail=tail, nu1=nu[0], nu2=nu[1], coarse_max_cells=2048)
            p = torch.zeros_like(rhs)
            for _ in range(2):
                ctx.vcycle(rhs, p)
            out.append(p)
        assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1]), prec


@pytest.mark.parametrize("shape", [(264, 16, 16), (320, 24, 16), (72, 24, 40), (256, 16, 32), (8, 16, 16)])
def test_row_blocks_identical_to_natural_layout(mgp, shape):
    """The finest colour passes, restriction and prolongation with rows that do and do not fill their
    blocks' rows of 32 threads: bit for bit the cycle on the natural layout (fused sweeps)."""
    case = synth.small_case(*shape, solid="ellipsoid", seed=53)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = dev(case.rhs)
    out = []
    for sm in (1, 2):
        ctx = mgp.Context(beta, case.h, prec="mixed", smoother=sm, coarse_max_cells=2048)
        p = torch.zeros_like(rhs)
        for _ in range(2):
            ctx.vcycle(rhs, p)
        out.append(p)
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("shape,stretched", [((48, 16, 24), False), ((36, 32, 32), False), ((64, 32, 32), True),
                                             ((10, 16, 16), True)])
def test_fp64_row_records_identical_to_loaded_faces(mgp, shape, stretched):
    """FP64 colour passes that take a row's faces and inverse diagonals from its record, uniform or
    one value per kind of face (a grid stretched in z): bit for bit the fused sweeps, which load every
    face."""
    nx, ny, nz = shape
    case = synth.small_case(nx, ny, nz, solid="ellipsoid", interface="flat", seed=54)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    h, area = case.h, None
    if stretched:
        w = [dev(np.full(nx, h)), dev(np.full(ny, h)), dev(synth.stretched_widths(nz))]
        beta, area = mgp.stretched_metrics(*w, beta)
        h = 1.0
    rhs = dev(case.rhs)
    out = []
    for sm in (1, 2):
        ctx = mgp.Context(beta, h, smoother=sm, coarse_max_cells=2048)
        ctx.set_face_areas(area)
        p = torch.zeros_like(rhs)
        for _ in range(2):
            ctx.vcycle(rhs, p)
        out.append(p)
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("nu,inner", [((2, 2), 1), ((1, 1), 2), ((0, 2), 1), ((5, 1), 1)])
@pytest.mark.parametrize("shape", [(48, 16, 24), (32, 32, 32), (16, 16, 16), (20, 16, 24)])
def test_passes_queued_ahead_change_nothing(mgp, shape, nu, inner):
    """A profiled solve queues every cycle after the host has read the residual before it; else
    the first passes are queued while the host waits.  The kernels and their order are the same:
    every bit agrees, iteration counts included, also where the cycle limit ends the solve."""
    for prec, cycles in (("fp64", 100), ("mixed", 100), ("mixed", 3)):
        got = []
        for profile in (0, 1):
            _, _, b, ctx = _setup(mgp, shape, prec=prec, krylov=1, nu1=nu[0], nu2=nu[1], inner_cycles=inner,
                                  max_cycles=cycles, profile=profile)
            p, st = ctx.solve(dev(b), tol=1e-10, allow_not_converged=True)
            got.append((host(p), st.cycles, st.rel_resid))
        assert got[0][1:] == got[1][1:], prec
        assert np.array_equal(got[0][0], got[1][0]), prec


@pytest.mark.parametrize("nu", [(2, 2), (3, 1), (1, 2), (2, 0)])
@pytest.mark.parametrize("shape", [(64, 48, 40), (36, 32, 32), (128, 16, 32), (20, 16, 24), (64, 64, 64)])
def test_joined_coarse_passes_identical_to_fused_sweeps(mgp, shape, nu):
    """Coarse levels whose first red and black passes, and whose prolongation and the black pass after
    it, are one launch each: bit for bit the fused sweeps, which store every red value between."""
    case = synth.small_case(*shape, solid="ellipsoid", seed=55)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = dev(case.rhs)
    for prec in ("fp64", "mixed"):
        out = []
        for sm in (1, 2):
            ctx = mgp.Context(beta, case.h, prec=prec, smoother=sm, coarse_max_cells=2048, coarse_tail=0, nu1=nu[0],
                              nu2=nu[1])
            p = torch.zeros_like(rhs)
            for _ in range(2):
                ctx.vcycle(rhs, p)
            out.append(p)
        assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1]), prec


@pytest.mark.parametrize("prec,shape", [("fp64", (256, 256, 256)), ("mixed", (448, 256, 256))])
def test_coarse_row_records_identical_to_loaded_faces(mgp, prec, shape):
    """Coarse levels large enough for row records (2.1 M cells in FP64, 3.7 M in FP32), with rows that
    have one and rows that have none: bit for bit the fused sweeps, which load every face."""
    nx, ny, nz = shape
    x, z = torch.linspace(0.0, 1.0, nx, device="cuda"), torch.linspace(0.0, 1.0, nz, device="cuda")
    phi = torch.sigmoid(40.0 * (0.5 + 0.1 * torch.sin(9.0 * x)[None, None, :] - z[:, None, None])).double()
    phi = phi.expand(nz, ny, nx).contiguous()
    phi[phi < 1e-3], phi[phi > 1 - 1e-3] = 0.0, 1.0
    beta = mgp.face_coeffs(phi, 1.0 / nx, None, rho_air=1e-3)
    g = torch.Generator(device="cuda").manual_seed(56)
    rhs = torch.randn(phi.shape, dtype=torch.float64, device="cuda", generator=g)
    rhs -= rhs.mean()
    out = []
    for sm in (1, 2):
        ctx = mgp.Context(beta, 1.0 / nx, prec=prec, smoother=sm)
        p = torch.zeros_like(rhs)
        for _ in range(2):
            ctx.vcycle(rhs, p)
        out.append(p)
        ctx.close()
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (3, 0), (1, 0)])
@pytest.mark.parametrize("shape", [(48, 16, 24), (32, 32, 32), (20, 16, 24)])
def test_stationary_passes_queued_ahead_change_nothing(mgp, shape, nu):
    """As above for the stationary cycles, whose passes ahead work on p itself and must store nothing
    once the iteration has ended: by its tolerance, its cycle limit or a residual that is not finite."""
    for prec, inner, cycles, tol, every in (("fp64", 1, 100, 1e-9, 1), ("fp64", 1, 100, 1e-5, 2), ("fp64", 1, 4, 1e-12, 1),
                                            ("mixed", 1, 100, 1e-9, 1), ("mixed", 2, 3, 1e-12, 1)):
        got = []
        for profile in (0, 1):
            _, _, b, ctx = _setup(mgp, shape, prec=prec, krylov=0, nu1=nu[0], nu2=nu[1], inner_cycles=inner,
                                  max_cycles=cycles, check_every=every, profile=profile)
            p, st = ctx.solve(dev(b), tol=tol, allow_not_converged=True)
            got.append((host(p), st.cycles, st.rel_resid))
        assert got[0][1:] == got[1][1:], (prec, tol)
        assert np.array_equal(got[0][0], got[1][0]), (prec, tol)
    out = []
    for profile in (0, 1):
        _, _, b, ctx = _setup(mgp, shape, krylov=0, nu1=nu[0], nu2=nu[1], profile=profile)
        p = dev(b * 1e200)  # a guess whose residual norm overflows
        with pytest.raises(mgp.MGError):
            ctx.solve(dev(b), p, tol=1e-9)
        out.append(host(p))
    assert np.array_equal(out[0], out[1], equal_nan=True)
