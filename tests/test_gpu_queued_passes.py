"""Passes queued ahead of the host's decision, and whether the paths that the bit-for-bit comparisons of the
cycle's passes compare are the ones that run."""
import numpy as np
import pytest
import torch

from paper_1410_2240_gb300 import synth

from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mgp():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_2240_gb300 import mgproj
    return mgproj


@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (3, 1), (1, 2), (2, 0), (1, 0)])
@pytest.mark.parametrize("shape", [(16, 16, 16), (48, 16, 24)])
def test_passes_queued_ahead_of_an_overflow_store_nothing(mgp, shape, nu):
    """Strong faces inside the coarse cells, which the coarse grids do not see: the first cycle from zero multiplies
    a random residual by 96 to 2900 (1e4 times stronger faces, the oracle's cycle).  With ||b||^2 = 1e306 the squared residual is finite before
    that cycle and overflows after it, when the next cycle's first passes are queued already; p is then the first cycle's, as
    in a profiled solve, which queues nothing ahead."""
    nx, ny, nz = shape
    beta = [np.ones((nz, ny, nx)) for _ in range(3)]
    for axis, b in zip((2, 1, 0), beta):
        at = [slice(None)] * 3
        at[axis] = slice(1, None, 2)
        b[tuple(at)] = 1e4
        at[axis] = 0
        b[tuple(at)] = 0.0
    rhs = np.random.default_rng(7).standard_normal((nz, ny, nx))
    rhs -= rhs.mean()
    rhs *= 1e153 / np.linalg.norm(rhs)
    out = []
    for profile in (0, 1):
        ctx = mgp.Context(tuple(dev(b) for b in beta), 1.0 / 16, nu1=nu[0], nu2=nu[1], profile=profile)
        p = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
        with pytest.raises(mgp.MGError, match="not finite after 1 cycles") as e:
            ctx.solve(dev(rhs), p, tol=1e-9)
        assert e.value.code == mgp.MG_ERR_NAN
        out.append(host(p))
    assert np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0.0
    assert np.array_equal(out[0], out[1])


def _rows(ctx, level):
    """Interior rows with one value on the x-, y-, low z- and high z-faces each, and the others."""
    bx, by, bz = (host(ctx.level_array(level, a)) for a in range(3))
    one = lambda a: (a == a[:, :, :1]).all(axis=2) & (a[:, :, 0] > 0)
    x = (bx[:, :, 1:] == bx[:, :, 1:2]).all(axis=2) & (bx[:, :, 1] > 0)
    y = one(by)[:, :-1] & one(by)[:, 1:] & (by[:, :-1, 0] == by[:, 1:, 0])
    z = one(bz)[:-1] & one(bz)[1:]
    ok = x[1:-1, 1:-1] & y[1:-1, 1:] & z[1:, 1:-1]
    return int(ok.sum()), int((~ok).sum())


@pytest.mark.parametrize("shape,stretched", [((48, 16, 24), False), ((36, 32, 32), False), ((64, 32, 32), True),
                                             ((10, 16, 16), True)])
def test_inputs_have_rows_with_and_without_a_record(mgp, shape, stretched):
    """The inputs on which the FP64 passes with row records are compared with those that load every face."""
    nx, ny, nz = shape
    case = synth.small_case(nx, ny, nz, solid="ellipsoid", interface="flat", seed=54)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    h, area = case.h, None
    if stretched:
        w = [dev(np.full(nx, h)), dev(np.full(ny, h)), dev(synth.stretched_widths(nz))]
        beta, area = mgp.stretched_metrics(*w, beta)
        h = 1.0
    ctx = mgp.Context(beta, h, coarse_max_cells=2048)
    ctx.set_face_areas(area)
    with_record, without = _rows(ctx, 0)
    assert with_record > 0 and without > 0


# first tail level (half the grid): planes left over on the last CTA, more cells of a colour per CTA than threads, CTAs
# without a plane, the largest tail, a coarsest grid of an odd size
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(32, 32, 40), (16, 16, 100), (40, 40, 40), (64, 32, 16), (32, 32, 64), (48, 16, 40),
                                   (20, 24, 28)])
def test_tail_runs_and_is_the_launches(mgp, shape, prec):
    """The coarse levels in one launch: fewer kernels than a launch per pass, the same bits."""
    case = synth.small_case(*shape, solid="ellipsoid", seed=52)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = dev(case.rhs)
    for nu in ((2, 2), (0, 1), (1, 0)):
        launches, out = [], []
        for tail in (0, 1):
            ctx = mgp.Context(beta, case.h, prec=prec, coarse_tail=tail, coarse_max_cells=2048, nu1=nu[0], nu2=nu[1])
            l0 = mgp.kernel_launches()
            p = torch.zeros_like(rhs)
            for _ in range(2):
                ctx.vcycle(rhs, p)
            out.append(p)
            launches.append(mgp.kernel_launches() - l0)
        assert launches[1] < launches[0]
        assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (2, 0)])
@pytest.mark.parametrize("prec,krylov,inner", [("fp64", 0, 1), ("mixed", 0, 2), ("fp64", 1, 2)])
def test_profiled_sweeps_are_whole_sweeps(mgp, prec, krylov, inner, nu):
    """Group 0 times sweeps of both colours: a cycle that continues another starts with a black pass alone
    (where it smooths on both ways), which is not one of them."""
    case = synth.small_case(48, 16, 24, solid="ellipsoid", seed=97)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = mgp.Context(beta, case.h, coarse_max_cells=2048).divergence(tuple(dev(u) for u in case.u_star))
    ctx = mgp.Context(beta, case.h, prec=prec, krylov=krylov, inner_cycles=inner, nu1=nu[0], nu2=nu[1], profile=1,
                      max_cycles=3, coarse_max_cells=2048)
    _, st = ctx.solve(rhs, tol=1e-30, allow_not_converged=True)
    assert st.cycles == 3
    sweeps, _ = ctx.profile_read(mgp.PROF_SMOOTH)
    cycles = 3 * (inner if prec == "mixed" or krylov else 1)
    continued = (2 if krylov == 0 and prec == "fp64" else 3 * (inner - 1)) if nu[1] else 0
    assert sweeps == cycles * sum(nu) - continued
