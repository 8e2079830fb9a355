"""The norms of hhg_residual, both parts in one launch, where the parts take one
block, different numbers of blocks, and more elements than blocks can hold once.

Tolerance: sums of n <= 2^24 squares in FP64, any order: n 2^-53 < 2e-9 at worst;
in blocks of at most 2^14 terms a chain 2e-12.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("disc,box,L", [("P1P1", (1, 1, 1), 1), ("P1P1", (1, 3, 2), 4), ("P2P1", (1, 1, 1), 2),
                                        ("P2P1", (2, 1, 1), 5)])
def test_norms_of_both_parts(disc, box, L, prec):
    from paper_2010_13513_gb300 import hhg
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    pb = hhg.Problem(hhg.Mesh.box(*box, 1.0 / max(box)), disc=disc, L=L, coarse_level=0 if disc == "P1P1" else 1,
                     solve="mixed")
    x, b, r = (pb.new_vector(L, p) for _ in range(3))
    n = x.numel()
    b.copy_(torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)))
    nu, npr = pb.residual(L, x, b, r, norms=True)
    n_u = n - n // (25 if disc == "P2P1" else 4)
    for got, part in ((nu, r[:n_u]), (npr, r[n_u:])):
        ref = float(part.double().norm())
        assert abs(got - ref) <= 2e-12 * ref
