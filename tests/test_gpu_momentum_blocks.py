"""The momentum terms where their blocks end: rows of more than one block, rows and planes left over,
one-cell-wide axes, and the calls that leave terms out.  Bit for bit the oracle's R (the same
separately rounded operations in the same order), with h a power of two and not."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1410_2240_gb300 import synth

from _gpu_util import dev, faces_dev, faces_host

pytestmark = pytest.mark.gpu

SHAPES = [(300, 5, 20), (256, 3, 9), (33, 17, 8), (31, 1, 17), (2, 40, 3), (512, 2, 1), (64, 16, 16)]


@pytest.fixture(scope="module")
def mgp():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_2240_gb300 import mgproj
    return mgproj


@pytest.mark.parametrize("inv_re,convection", [(0.37, True), (0.37, False), (0.0, True), (0.0, False)])
@pytest.mark.parametrize("shape", SHAPES)
def test_momentum_blocks_bit_exact(mgp, shape, inv_re, convection):
    case = synth.small_case(*shape, seed=61, solid="none", interface="random")
    beta = O.face_coeffs(case.phi, None, case.lam)
    R_o = O.momentum_rhs(case.phi, beta, case.u_star, case.h, g=1.3, inv_re=inv_re, mu_air=1.8e-2, convect=convection)
    f = mgp.forces(g=1.3, inv_re=inv_re, mu_air=1.8e-2, convection=convection)
    R_g = mgp.momentum_rhs(dev(case.phi), faces_dev(beta), faces_dev(case.u_star), case.h, f)
    for a, b in zip(faces_host(R_g), R_o):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("shape", [(256, 40, 61), (256, 38, 64)])
def test_momentum_long_and_short_runs_bit_exact(mgp, shape):
    """160 blocks of eight planes (long runs) and 152 of them; one row pair less takes the short runs
    that the smaller shapes above take."""
    for sh in (shape, (shape[0], shape[1] - 2, shape[2])):
        test_momentum_blocks_bit_exact(mgp, sh, 0.37, True)
