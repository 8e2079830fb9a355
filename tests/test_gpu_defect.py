"""The unrolled double-float defect where its warps are ragged: planes below
64 positions (one site per lane), planes whose last warp starts early, boxes
that are no cubes (h not a power of two).

Tolerance: the documented bound of the double-float rows against an exact
evaluation, 2^-24 |r| + (n^2 2^-48 + 2^-46) sum_j |a_ij x_j| with n <= 238
terms (n^2 2^-48 < 2^-32), and b counted as one more term; the FP64 oracle's
own error is far below it.  b = calA x + 1e-6 noise, so that every row cancels.
"""
import numpy as np
import pytest

from gpu_helpers import lib_problem, oracle_hierarchy, random_vector
from test_gpu_parity import _abs_row_sums

pytestmark = pytest.mark.gpu


# the second line: levels above the sizes that keep the looped kernel
@pytest.mark.parametrize("disc,box,L", [("P1P1", (1, 1, 1), 1), ("P1P1", (3, 1, 2), 3), ("P2P1", (1, 1, 1), 1),
                                        ("P2P1", (3, 1, 1), 2), ("P2P1", (1, 2, 1), 3),
                                        ("P1P1", (3, 1, 2), 5), ("P2P1", (3, 1, 1), 4), ("P2P1", (1, 1, 42), 2)])
def test_defect_rows(disc, box, L):
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" or box[2] > 3 else 1
    pb = lib_problem(box, L, disc, lc=lc, solve="mixed")
    lev = oracle_hierarchy(box, L, disc, lc=lc).lv[L]
    assert pb.refinement_residual_kind() == "df32"
    x = random_vector(lev, 1)
    b = lev.apply(x) + 1e-6 * random_vector(lev, 2)
    ref = lev.residual(x, b)
    r = pb.new_vector(L, hhg.FP32)
    r.fill_(7.0)                                                     # every node is written
    pb.refinement_residual(L, pb.to_device(L, x), pb.to_device(L, b), r)
    bound = 2.0 ** -24 * np.abs(ref) + (2.0 ** -32 + 2.0 ** -46) * (_abs_row_sums(lev, x) + np.abs(b))
    err = np.abs(pb.to_host(L, r) - ref)
    assert np.all(err <= bound), float((err - bound).max())
