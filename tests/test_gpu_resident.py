"""The shared-memory-resident smoother against the oracle where its slabs and
slots are ragged: one cell planes, CTAs that own only the top plane, rows
shorter than a vertex quad, several passes of a CTA over its slots.

Tolerance: an Uzawa iteration in FP64 is held to 1e-12 relative, as the
per-phase kernels are; in FP32 the unit roundoff is 2^29 times larger, and the
iterates are held to 1e-12 * 2^29 = 5e-4.
"""
import numpy as np
import pytest

from gpu_helpers import OMEGA_INV, lib_problem, oracle_hierarchy, random_vector, rel

pytestmark = pytest.mark.gpu

CASES = [
    ("P1P1", (1, 1, 1), 1, 0.0, 3, 128),       # one interior vertex; the third CTA owns the top plane only
    ("P1P1", (3, 1, 2), 2, 0.0, 9, 128),
    ("P1P1", (1, 2, 1), 3, 1.7, 2, 1024),
    ("P2P1", (1, 1, 1), 2, 0.0, 1, 128),       # several slots per thread
    ("P2P1", (1, 1, 1), 2, 1.1, 5, 160),
    ("P2P1", (2, 1, 1), 2, 0.0, 4, 256),
    ("P2P1", (1, 1, 1), 3, 0.0, 8, 1024),
]
# levels that fit the compact layout only
COMPACT = [
    ("P1P1", (2, 3, 1), 4, 0.0, 16, 1024, "fp32"),
    ("P1P1", (1, 2, 3), 3, 1.7, 1, 256, "fp32"),
    ("P1P1", (1, 3, 1), 4, 0.0, 9, 512, "fp64"),
    ("P1P1", (3, 1, 1), 4, 1.2, 16, 1024, "fp64"),
    ("P2P1", (2, 2, 1), 3, 0.0, 5, 1024, "fp32"),
    ("P2P1", (1, 1, 1), 4, 0.9, 9, 512, "fp32"),
]


@pytest.mark.parametrize("ahat,xi", [("f", 3), ("s", 2)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("disc,box,L,nu_a,ctas,threads", CASES)
def test_resident_smoother(disc, box, L, nu_a, ctas, threads, prec, ahat, xi):
    check(disc, box, L, nu_a, ctas, threads, prec, ahat, xi)


@pytest.mark.parametrize("ahat,xi", [("f", 2), ("s", 1)])
@pytest.mark.parametrize("disc,box,L,nu_a,ctas,threads,prec", COMPACT)
def test_compact_layout(disc, box, L, nu_a, ctas, threads, prec, ahat, xi):
    check(disc, box, L, nu_a, ctas, threads, prec, ahat, xi)


def check(disc, box, L, nu_a, ctas, threads, prec, ahat, xi):
    from oracle.stokes import Params
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, nu_a=nu_a, solve="mixed")
    lev = oracle_hierarchy(box, L, disc, lc=lc, nu_a=nu_a).lv[L]
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    pb.set_level_smoother(L, ctas, threads, p)
    x, b = random_vector(lev, 1), random_vector(lev, 2)
    xd, bd = pb.to_device(L, x, p), pb.to_device(L, b, p)
    om = OMEGA_INV[disc]
    pb.smooth(L, hhg.Params.make(1, 1, 0, 1, ahat, xi, om), 2, xd, bd)
    prm = Params(1, 1, 0, 1, ahat, xi, om)
    ref = lev.uzawa(lev.uzawa(x, b, prm), b, prm)
    assert rel(pb.to_host(L, xd), ref) < (1e-12 if prec == "fp64" else 5e-4)
