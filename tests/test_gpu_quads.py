"""B^T and the pressure step on large P1-P1 levels: four aligned sites per
thread against a site per thread, which takes vectors that are not 16-byte
aligned.

Tolerance: two FP32 evaluations of a row of at most 60 terms differ by at most
2 * 60 * 2^-24 = 7.2e-6 of sum |a_j x_j|, for random x about sqrt(60) times the
row's value: 6e-5 of the row, and an Uzawa iteration is of the size of its rows.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu_a", [0.0, 1.3])
@pytest.mark.parametrize("box", [(2, 2, 1), (1, 3, 2)])
def test_aligned_quads_match_single_sites(box, nu_a):
    from paper_2010_13513_gb300 import hhg
    L = 7
    pb = hhg.Problem(hhg.Mesh.box(*box, 1.0 / max(box)), disc="P1P1", L=L, coarse_level=1, solve="mixed", nu_a=nu_a)
    pb.set_level_smoother(L, 0)
    n = pb.new_vector(L, hhg.FP32).numel()
    nx, ny, nz = (c << L for c in box)
    sx = (nx + 6) // 4 * 4
    rng = torch.Generator(device="cuda").manual_seed(3)

    def lattice(dirichlet):
        v = torch.zeros(4, n // 4, device="cuda")
        q = v[:, :sx * (ny + 3) * (nz + 3)].unflatten(1, (nz + 3, ny + 3, sx))
        q[:, 1:nz + 2, 1:ny + 2, 1:nx + 2] = torch.randn(4, nz + 1, ny + 1, nx + 1, device="cuda", generator=rng)
        if dirichlet:
            inner = q[:3, 2:nz + 1, 2:ny + 1, 2:nx + 1].clone()
            q[:3] = 0
            q[:3, 2:nz + 1, 2:ny + 1, 2:nx + 1] = inner
        return v.flatten()

    x, b = lattice(True), lattice(False)
    buf = torch.zeros(n + 4, device="cuda")
    shifted = buf[1:1 + n]
    shifted.copy_(x)
    prm = hhg.Params.make(1, 1, 0, 1, "f", 1, 0.5)
    pb.smooth(L, prm, 1, x, b)
    pb.smooth(L, prm, 1, shifted, b)
    torch.cuda.synchronize()
    for part in (slice(0, 3 * (n // 4)), slice(3 * (n // 4), n)):
        err = (x[part].double() - shifted[part].double()).norm() / shifted[part].double().norm()
        assert float(err) < 6e-5
    pad = x.view(4, -1)[:, :sx * (ny + 3) * (nz + 3)].unflatten(1, (nz + 3, ny + 3, sx))
    assert not pad[:, 0].any() and not pad[:, :, 0].any() and not pad[..., 0].any() and not pad[..., nx + 2:].any()
