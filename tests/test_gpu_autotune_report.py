"""hhg_autotune reports the launch shapes that the smoother's B^T and (B, -C) rows
run with: several planes per block above a million sites, four sites per thread
above four million (P1-P1 in FP32)."""
import pytest

from gpu_helpers import lib_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc,box,L,solve,bt,bc", [
    ("P1P1", (2, 2, 1), 6, "mixed", (128, 1, 1), (256, 4, 1)),       # 1.1 million sites
    ("P1P1", (4, 2, 2), 6, "mixed", (256, 4, 4), (256, 4, 4)),       # 4.3 million
    ("P1P1", (4, 2, 2), 6, "fp64", (128, 1, 1), (256, 4, 1)),
    ("P2P1", (2, 2, 1), 6, "mixed", (128, 1, 1), (256, 4, 1)),
])
def test_shapes(disc, box, L, solve, bt, bc):
    pb = lib_problem(box, L, disc, lc=0 if disc == "P1P1" else 1, solve=solve)
    shapes = pb.autotune(reps=1)
    assert shapes[L][9:12] == bt and shapes[L][12:15] == bc
    assert shapes[3][9:15] == (128, 1, 1, 256, 1, 1)
