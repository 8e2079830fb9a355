"""The smoother's separate launches (no shared-memory-resident level) against
the oracle, where their tiles and runs are ragged: planes just wider than a
tile, runs of two planes, odd numbers of passes, levels smaller than a halo.

Tolerance: an Uzawa iteration in FP64 is held to 1e-12 relative; in FP32 the
unit roundoff is 2^29 times larger: 1e-12 * 2^29 = 5e-4.
"""
import pytest

from gpu_helpers import OMEGA_INV, lib_problem, oracle_hierarchy, random_vector, rel

pytestmark = pytest.mark.gpu

CASES = [
    ("P1P1", (1, 1, 1), 1, 0.0),
    ("P1P1", (1, 1, 3), 2, 0.0),
    ("P1P1", (3, 1, 2), 5, 0.0),               # 97 x 33 x 65 sites: two tiles (FP64: four) in i
    ("P1P1", (1, 2, 1), 4, 1.7),
    ("P2P1", (1, 1, 1), 1, 0.0),
    ("P2P1", (3, 1, 1), 3, 0.0),
    ("P2P1", (1, 2, 1), 3, 1.1),
    ("P2P1", (1, 1, 1), 4, 0.0),
]


@pytest.mark.parametrize("ahat,xi", [("f", 1), ("f", 2), ("s", 1)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("disc,box,L,nu_a", CASES)
def test_separate_launches(disc, box, L, nu_a, prec, ahat, xi):
    from oracle.stokes import Params
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, nu_a=nu_a, solve="mixed")
    lev = oracle_hierarchy(box, L, disc, lc=lc, nu_a=nu_a).lv[L]
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    pb.set_level_smoother(L, 0, prec=p)
    x, b = random_vector(lev, 1), random_vector(lev, 2)
    om = OMEGA_INV[disc]
    prm = Params(1, 1, 0, 1, ahat, xi, om)
    ref = lev.uzawa(lev.uzawa(x, b, prm), b, prm)
    for order in (0, 1):
        pb.set_sweep_order(L, order)
        xd, bd = pb.to_device(L, x, p), pb.to_device(L, b, p)
        pb.smooth(L, hhg.Params.make(1, 1, 0, 1, ahat, xi, om), 2, xd, bd)
        assert rel(pb.to_host(L, xd), ref) < (1e-12 if prec == "fp64" else 5e-4), order
