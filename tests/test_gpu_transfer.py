"""The unrolled transfer kernels against the oracle on boxes whose planes span
several ragged blocks, in both precisions.

Tolerance: every output is a sum of at most 130 products whose weights' moduli
add up to less than 16, so it is off by at most 130 * u * 16 * max|x| (u the
unit roundoff of the precision), plus one rounding of the updated value.
"""
import numpy as np
import pytest

from gpu_helpers import lib_problem, oracle_hierarchy, random_vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("disc,box,L", [("P1P1", (1, 1, 1), 1), ("P1P1", (3, 1, 2), 3), ("P2P1", (1, 1, 1), 2),
                                        ("P2P1", (3, 2, 1), 3)])
def test_transfers(disc, box, L, prec):
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, solve="mixed")
    hy = oracle_hierarchy(box, L, disc, lc=lc)
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    cast = (lambda a: a) if prec == "fp64" else (lambda a: a.astype(np.float32).astype(np.float64))
    for l in range(lc + 1, L + 1):
        xf = cast(random_vector(hy.lv[l], 1, zero_dirichlet=False))      # Dirichlet entries must stay
        xc = cast(random_vector(hy.lv[l - 1], 2))
        d = pb.to_device(l, xf, p)
        pb.prolongate_add(l, pb.to_device(l - 1, xc, p), d)
        tol = 130 * 16 * u * max(np.abs(xf).max(), np.abs(xc).max())
        assert np.abs(pb.to_host(l, d) - (xf + hy.prolongate(l, xc))).max() <= tol
        rf = cast(random_vector(hy.lv[l], 3))
        rc = pb.new_vector(l - 1, p)
        rc.fill_(7.0)                                                    # every node is written
        pb.restrict(l, pb.to_device(l, rf, p), rc)
        assert np.abs(pb.to_host(l - 1, rc) - hy.restrict(l, rf)).max() <= tol
