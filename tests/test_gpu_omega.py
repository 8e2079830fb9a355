"""The spectral estimate of the pressure step (power iteration) against the
oracle on boxes with ragged planes: its rows B u - C p run in a kernel of their
own.  Tolerance as for the cube: 1e-10 relative after 30 iterations in FP64.
"""
import numpy as np
import pytest

from gpu_helpers import lib_problem, oracle_hierarchy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc,box,L,nu_a", [("P1P1", (1, 1, 1), 1, 0.0), ("P1P1", (3, 1, 2), 3, 0.0),
                                             ("P1P1", (3, 2, 1), 3, 1.3), ("P2P1", (1, 1, 1), 1, 0.0),
                                             ("P2P1", (3, 1, 2), 2, 0.0), ("P2P1", (1, 2, 1), 3, 1.1)])
def test_estimate(disc, box, L, nu_a):
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, nu_a=nu_a)
    hy = oracle_hierarchy(box, L, disc, lc=lc, nu_a=nu_a)
    v0 = np.random.default_rng(0).uniform(-1, 1, hy.lv[L].np)
    assert abs(pb.estimate_omega(L, v0, iters=30) / hy.estimate_omega_inv(v0, iters=30) - 1) < 1e-10
