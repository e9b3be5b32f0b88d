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


def _beta(mgp, shape=(16, 16, 16), solid="ellipsoid"):
    case = synth.small_case(*shape, solid=solid, seed=61)
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
