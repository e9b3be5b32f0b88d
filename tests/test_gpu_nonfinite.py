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


@pytest.mark.parametrize("areas,body", [(False, False), (True, False), (False, True), (True, True)])
def test_divergence_of_zeros_of_either_sign(mgp, areas, body):
    """The sum over a cell's faces starts from +0, so velocities that are zeros of either sign give the
    zeros that the six additions and subtractions give, sign for sign."""
    case, beta = _beta(mgp)
    rng = np.random.default_rng(62)
    zeros = lambda: np.where(rng.random(case.phi.shape) < 0.5, 0.0, -0.0)
    u, v = [zeros() for _ in range(3)], [zeros() for _ in range(3)]
    ctx = mgp.Context(beta, case.h)
    if areas:
        ctx.set_face_areas(tuple(dev(np.full(case.phi.shape, 0.5)) for _ in range(3)))
    if body:
        ctx.set_body_velocity(tuple(dev(x) for x in v))
    got = host(ctx.divergence(tuple(dev(x) for x in u)))
    d = np.zeros(case.phi.shape)
    for axis, b, x, y in zip((2, 1, 0), beta, u, v):
        flux = x - y if body else x
        at = lambda a, lo, hi: a[tuple(slice(lo, hi) if i == axis else slice(None) for i in range(3))]
        is_open, f = host(b) > 0, flux
        at(d, 0, -1)[...] = np.where(at(is_open, 1, None), at(d, 0, -1) + at(f, 1, None), at(d, 0, -1))
        d = np.where(is_open, d - f, d)
    assert np.array_equal(got, d) and np.array_equal(np.signbit(got), np.signbit(d))


@pytest.mark.parametrize("shape", [(16, 12, 20), (104, 100, 100)])
def test_stretched_metrics_divide_closed_faces_too(mgp, shape):
    """Widths are not checked: 0 / d on a closed face is the quotient, NaN or a zero of either sign, whatever d is."""
    nx, ny, nz = shape
    rng = np.random.default_rng(63)
    widths = [rng.choice([0.5, 1.0, 0.0, -1.0, float("nan")], n) for n in shape]
    beta = [np.where(rng.random((nz, ny, nx)) < 0.5, 0.0, 2.0) for _ in range(3)]
    got, area = mgp.stretched_metrics(*(dev(w) for w in widths), tuple(dev(b) for b in beta))
    for a, (b, g) in enumerate(zip(beta, got)):
        d = 0.5 * (widths[a][:-1] + widths[a][1:])
        want = np.zeros_like(b)
        inner = [slice(None)] * 3
        inner[2 - a] = slice(1, None)
        with np.errstate(all="ignore"):
            want[tuple(inner)] = b[tuple(inner)] / d.reshape([-1 if i == 2 - a else 1 for i in range(3)])
        g = host(g)
        assert np.array_equal(g, want, equal_nan=True), a
        number = ~np.isnan(want)
        assert np.array_equal(np.signbit(g[number]), np.signbit(want[number])), a
