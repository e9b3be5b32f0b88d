"""Coefficients and velocities at the edge of arithmetic: NaN and infinite face coefficients, zeros of either
sign.  What is compared is exact (an error code, a bit pattern), so there are no bounds."""
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


def _beta(mgp):
    case = synth.small_case(16, solid="ellipsoid", seed=61)
    return case, mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_operator_that_is_not_finite_is_refused(mgp, prec, axis, bad):
    """A NaN or an infinity on a face of the coarsest grid (every fourth one here) makes its operator one that
    has no inverse: an argument error from the set-up and from an update, after which the context
    still takes a finite operator."""
    case, beta = _beta(mgp)
    broken = [b.clone() for b in beta]
    at = [1, 2, 3]
    at[2 - axis] = 4
    broken[axis][tuple(at)] = bad
    with pytest.raises(mgp.MGError) as e:
        mgp.Context(tuple(broken), case.h, prec=prec)
    assert e.value.code == mgp.MG_ERR_ARG
    ctx = mgp.Context(beta, case.h, prec=prec)
    rhs = dev(case.rhs)
    want = host(ctx.vcycle(rhs, torch.zeros_like(rhs)))
    with pytest.raises(mgp.MGError) as e:
        ctx.update(tuple(broken))
    assert e.value.code == mgp.MG_ERR_ARG
    ctx.update(beta)
    assert np.array_equal(host(ctx.vcycle(rhs, torch.zeros_like(rhs))), want)


@pytest.mark.parametrize("krylov", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_nan_between_coarse_faces_leaves_its_cells_without_a_diagonal(mgp, prec, krylov):
    """A NaN on a face that no coarse level sees: the diagonal of its two cells is no positive number, so their
    inverse is 0 (as for cells without an open face), every other one stands, and a solve reports NaN."""
    case, beta = _beta(mgp)
    want = host(mgp.Context(beta, case.h, prec=prec).level_array(0, 3))
    beta[0][2, 3, 5] = float("nan")
    ctx = mgp.Context(beta, case.h, prec=prec, krylov=krylov)
    want[2, 3, 4:6] = 0.0
    assert np.array_equal(host(ctx.level_array(0, 3)), want)
    with pytest.raises(mgp.MGError) as e:
        ctx.solve(dev(case.rhs))
    assert e.value.code == mgp.MG_ERR_NAN
