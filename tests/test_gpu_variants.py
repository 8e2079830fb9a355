"""Kernel variants that the dispatch takes on large or wide levels only: the
prolongation in aligned pairs (even pitch: nx >= 64), the vertex colours on shared
edge sums (P2-P1 above a million sites) and the marching rows with a variable
viscosity.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import curl_workload, lib_problem, oracle_hierarchy, random_vector, rel
from test_gpu_fullsize import EPS32, _dirichlet_mask, _gather, _pick_rows

pytestmark = pytest.mark.gpu


def outside(pb, level, v):
    """The elements of a device vector that are no node."""
    info = pb.layout(level)
    ones = np.ones(3 * info.n_velocity_nodes + info.n_pressure_nodes)
    return v[pb.to_device(level, ones) == 0]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("disc,box,L", [("P1P1", (4, 1, 1), 4), ("P1P1", (5, 1, 2), 4), ("P2P1", (4, 1, 1), 4),
                                        ("P2P1", (5, 1, 1), 4)])
def test_prolongation_in_pairs(disc, box, L, prec):
    """nx = 64 (the row ends two sites before the pitch) and 80, against the
    oracle; a target shifted by one element, which takes single sites, gives the
    same bits.  Tolerance: a value is a sum of at most ten products whose weights'
    moduli add up to at most 5/2, and is added to the old one: 12 roundings of at
    most 3.5 max|x|."""
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, solve="mixed")
    hy = oracle_hierarchy(box, L, disc, lc=lc)
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    cast = (lambda a: a) if prec == "fp64" else (lambda a: a.astype(np.float32).astype(np.float64))
    xf = cast(random_vector(hy.lv[L], 1, zero_dirichlet=False))       # Dirichlet entries must stay
    xc = cast(random_vector(hy.lv[L - 1], 2))
    d, c = pb.to_device(L, xf, p), pb.to_device(L - 1, xc, p)
    shifted = torch.empty(d.numel() + 1, dtype=d.dtype, device=d.device)[1:]
    shifted.copy_(d)
    pb.prolongate_add(L, c, d)
    pb.prolongate_add(L, c, shifted)
    torch.cuda.synchronize()
    assert torch.equal(d, shifted)
    assert outside(pb, L, d).abs().max() == 0
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    assert np.abs(pb.to_host(L, d) - (xf + hy.prolongate(L, xc))).max() <= 12 * u * 3.5


@pytest.mark.parametrize("disc,L,s", [("P1P1", 4, (2, 2, 1, 1, "s", 1)), ("P2P1", 4, (1, 1, 0, 1, "f", 2))])
def test_fmg_start_values_in_pairs(disc, L, s):
    """FMG on 4 x 1 x 1 cubes: its last stage starts from the interpolation that
    sets the fine vector (in pairs).  Tolerance as for the FMG on the other boxes."""
    from oracle.stokes import Params
    from paper_2010_13513_gb300 import hhg
    lc, om = (0, 0.5) if disc == "P1P1" else (1, 0.3)
    wl = curl_workload()
    pb = lib_problem((4, 1, 1), L, disc, lc=lc, workload=wl)
    x = pb.new_vector(L)
    pb.fmg_solve(hhg.Params.make(*s, om), x, stats=False)
    ref = oracle_hierarchy((4, 1, 1), L, disc, lc=lc, workload=wl).fmg(Params(*s, om))
    assert rel(pb.to_host(L, x), ref) < 1e-10
    assert outside(pb, L, x).abs().max() == 0


@pytest.mark.parametrize("ahat,xi", [("f", 2), ("s", 1)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nu_a", [0.0, 1.3])
def test_shared_edge_sums(nu_a, prec, ahat, xi):
    """193 x 65 x 129 sites, ragged tiles and plane groups: the vertex colours on
    shared edge sums (the default order there) against the component order, whose
    full rows the oracle checks on small levels.  The same iterates up to
    rounding: 1e-12 in FP64, 2^29 times as much in FP32."""
    from paper_2010_13513_gb300 import hhg
    L = 6
    pb = lib_problem((3, 1, 2), L, "P2P1", lc=1, nu_a=nu_a, solve="mixed")
    p = hhg.FP64 if prec == "fp64" else hhg.FP32
    pb.set_level_smoother(L, 0, prec=p)
    assert pb.sweep_order(L) == 0
    info = pb.layout(L)
    n = 3 * info.n_velocity_nodes + info.n_pressure_nodes
    rng = np.random.default_rng(3)
    x, b = rng.uniform(-1.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    x[:3 * info.n_velocity_nodes] *= np.tile(~_dirichlet_mask(info, "P2P1"), 3)
    bd, out = pb.to_device(L, b, p), []
    for order in (0, 1):
        pb.set_sweep_order(L, order)
        xd = pb.to_device(L, x, p)
        pb.smooth(L, hhg.Params.make(1, 1, 0, 1, ahat, xi, 0.3), 1, xd, bd)
        torch.cuda.synchronize()
        out.append(xd)
    assert outside(pb, L, out[0]).abs().max() == 0
    d = (out[0].double() - out[1].double()).norm() / out[1].double().norm()
    assert 0 < d < (1e-12 if prec == "fp64" else 1e-12 * 2 ** 29)    # (0: the same kernels)


def test_marching_rows_with_variable_viscosity():
    """129 x 129 x 65 sites, sampled rows against the oracle (tolerance of the
    full-size rows: 256 eps s)."""
    from oracle.sampled import sample_rows
    from paper_2010_13513_gb300 import hhg
    box, H, L, nu_a = (2, 2, 1), 0.5, 6, 1.3
    pb = hhg.Problem(hhg.Mesh.box(*box, H), disc="P2P1", L=L, coarse_level=1, solve="mixed", nu_a=nu_a)
    info = pb.layout(L)
    nv = info.n_velocity_nodes
    rng = np.random.default_rng(11)
    n = 3 * nv + info.n_pressure_nodes
    x, b = (rng.uniform(-1.0, 1.0, n).astype(np.float32).astype(np.float64) for _ in range(2))
    for v in (x, b):
        v[:3 * nv] *= np.tile(~_dirichlet_mask(info, "P2P1"), 3)
    rows = _pick_rows((info.nx, info.ny, info.nz), "P2P1", rng, per_kind=2)
    ref, s = sample_rows(box, H, L, "P2P1", x, rows, nu_a, with_abs=True)
    xd, y = pb.to_device(L, x, hhg.FP32), pb.new_vector(L, hhg.FP32)
    pb.apply(L, "FULL", xd, y)
    got = _gather(pb.to_host(L, y), rows, nv)
    assert np.all(np.abs(got - ref) <= 256 * EPS32 * s) and np.all(got[s == 0.0] == 0.0)
    pb.residual(L, xd, pb.to_device(L, b, hhg.FP32), y)
    brow = _gather(b, rows, nv)
    assert np.all(np.abs(_gather(pb.to_host(L, y), rows, nv) - (brow - ref)) <= 256 * EPS32 * (s + np.abs(brow)))
