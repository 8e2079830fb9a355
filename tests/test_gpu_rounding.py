"""FP32 rounding errors of the kernels' sums against those of plain sums of the
same terms, both against 64 bits.

A plain sum is emulated in numpy: the products of FP32 numbers are exact in 64
bits, so fma(w, x, a) is one rounding of the 64-bit value to FP32.  A kernel may
order and split a row as it likes, but its error (root mean square over the
rows) is no larger than that of the plain sum.
"""
import numpy as np
import pytest

from gpu_helpers import OMEGA_INV, lib_problem, oracle_hierarchy, random_vector

pytestmark = pytest.mark.gpu

F = np.float32


def f32(a):
    return np.asarray(a, dtype=np.float64).astype(F).astype(np.float64)


def plain_sum(w, x, chains=1):
    """Rows of terms (rows x terms) summed in FP32 by `chains` chains, to which
    the terms are dealt in turn; the chains are added up pairwise."""
    a = [np.zeros(x.shape[0], dtype=F) for _ in range(chains)]
    for t in range(x.shape[1]):
        a[t % chains] = (f32(w[:, t]) * x[:, t] + a[t % chains]).astype(F)
    while len(a) > 1:
        a = [a[i] + a[i + len(a) // 2] for i in range(len(a) // 2)]
    return a[0].astype(np.float64)


def rms(e):
    return float(np.sqrt(np.mean(np.square(e))))


def allowed(n):
    """Ratio of the root mean squares over n rows of two sums of the same error:
    each is known to 1 / sqrt(2 n)."""
    return 1 + 3 * np.sqrt(2 / (2 * n))


def by_length(R):
    """The rows of a sparse matrix by their number of terms: (rows, columns, weights)."""
    n = np.diff(R.indptr)
    for k in np.unique(n[n > 0]):
        rows = np.nonzero(n == k)[0]
        at = R.indptr[rows][:, None] + np.arange(k)
        yield rows, R.indices[at], R.data[at]


@pytest.mark.parametrize("disc,box,L", [("P1P1", (3, 1, 2), 4), ("P2P1", (3, 1, 2), 3)])
def test_restriction(disc, box, L):
    """A restriction row in eight chains (P1 fields: two) of equal length."""
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, solve="mixed")
    hy = oracle_hierarchy(box, L, disc, lc=lc)
    fine, coarse = hy.lv[L], hy.lv[L - 1]
    rf = f32(random_vector(fine, 3))
    rc = pb.new_vector(L - 1, hhg.FP32)
    pb.restrict(L, pb.to_device(L, rf, hhg.FP32), rc)
    (u, p), (cu, cp) = fine.split(rf), coarse.split(pb.to_host(L - 1, rc))
    for name, P, x, c, keep, chains in (("velocity", hy.Pv[L], u, cu, coarse.vint, 2 if disc == "P1P1" else 8),
                                        ("pressure", hy.Pp[L], [p], [cp], np.ones(coarse.np, bool), 2)):
        lib, plain = [], []
        for rows, cols, w in by_length(P.T.tocsr()):
            s = keep[rows]
            for xc, cc in zip(x, c):
                exact = (w[s] * xc[cols[s]]).sum(1)
                lib.append(cc[rows[s]] - exact)
                plain.append(plain_sum(w[s], xc[cols[s]], chains) - exact)
        lib, plain = np.concatenate(lib), np.concatenate(plain)
        print(f"{disc} {name}: {rms(lib):.3e}, plain {rms(plain):.3e}, ratio {rms(lib) / rms(plain):.3f}")
        assert rms(lib) <= allowed(lib.size) * rms(plain)


def sine_velocity(shape, seed=1):
    """Canonical velocity lattice (z, y, x) of sine modes that vanish on the
    boundary, with a tenth of noise: what a smoother meets."""
    rng = np.random.default_rng(seed)
    X = [np.linspace(0, 1, m) for m in shape]
    u = np.zeros((3,) + shape)
    for c in range(3):
        for _ in range(4):
            s = [np.sin(np.pi * rng.integers(1, 4) * x) for x in X]
            u[c] += rng.standard_normal() * s[0][:, None, None] * s[1][:, None] * s[2]
    u[:, 1:-1, 1:-1, 1:-1] += 0.1 * rng.standard_normal((3,) + tuple(m - 2 for m in shape))
    u[:, [0, -1]] = u[:, :, [0, -1]] = u[:, :, :, [0, -1]] = 0
    return f32(u)


def divergence_terms(disc):
    """An interior row of B at h = 1: (component, lattice offset x, y, z, weight)
    by component, group of the parity offset and cell offset (x slowest), and the
    row's lumped mass."""
    q = 2 if disc == "P2P1" else 1
    L, lc = 2, 0 if disc == "P1P1" else 1
    lev = oracle_hierarchy((1, 1, 1), L, disc, lc=lc).lv[L]
    n, h = 4, 0.25
    m, group = q * n + 1, {(0, 0, 0): 0, (1, 0, 0): 1, (0, 1, 0): 2, (0, 0, 1): 3, (1, 1, 0): 4, (1, 0, 1): 5,
                           (0, 1, 1): 6, (1, 1, 1): 7}
    row = (n // 2) * (1 + (n + 1) * (1 + (n + 1)))
    terms = []
    for c in range(3):
        B = lev.B[c].tocsr()
        for col, w in zip(B.indices[B.indptr[row]:B.indptr[row + 1]], B.data[B.indptr[row]:B.indptr[row + 1]]):
            d = np.array([col % m, col // m % m, col // (m * m)]) - q * n // 2
            if abs(w) > 1e-13 * abs(B.data).max():
                terms.append((c, group[tuple(d % q)], *(d // q), d, w / h ** 2))
    terms.sort(key=lambda t: t[:5])
    return [(t[0], *t[5], t[6]) for t in terms], lev.ML_hat[row] / h ** 3


@pytest.mark.parametrize("disc,L,path", [("P1P1", 5, "residual"), ("P1P1", 5, "separate"), ("P1P1", 5, "resident"),
                                         ("P2P1", 5, "residual"), ("P2P1", 5, "separate"), ("P2P1", 4, "resident")])
def test_pressure_row(disc, L, path):
    """B u of a smooth velocity, whose terms cancel: at most the error of one
    chain over the row.  In the smoother the row meets the velocity it has just
    written, and the factor omega M_L^-1 adds two roundings to both sides."""
    from paper_2010_13513_gb300 import hhg
    pb = lib_problem((1, 1, 1), L, disc, lc=0 if disc == "P1P1" else 1, solve="mixed")
    q, n = 2 if disc == "P2P1" else 1, 2 ** L
    vshape, npress = (q * n + 1,) * 3, (n + 1) ** 3
    nv = 3 * (q * n + 1) ** 3
    u = sine_velocity(vshape)
    xd = pb.to_device(L, np.concatenate([u.ravel(), np.zeros(npress)]), hhg.FP32)
    zero = pb.new_vector(L, hhg.FP32)
    terms, mass = divergence_terms(disc)
    h, om = 1.0 / n, OMEGA_INV[disc]
    if path == "residual":
        y = pb.new_vector(L, hhg.FP32)
        pb.residual(L, xd, zero, y)
        factor, out = -1.0, pb.to_host(L, y)
    else:
        pb.set_level_smoother(L, 0 if path == "separate" else 16, prec=hhg.FP32)
        pb.smooth(L, hhg.Params.make(1, 1, 0, 1, "f", 1, om), 1, xd, zero)
        out = pb.to_host(L, xd)
        factor = 1.0 / (om * mass * h ** 3)
        u = out[:nv].reshape((3,) + vshape)

    def at(c, dx, dy, dz):                         # the DoF at an offset from every interior pressure node
        s = [slice(q + d, q * (n - 1) + d + 1, q) for d in (dz, dy, dx)]
        return u[(c, *s)].ravel()

    X = np.stack([at(*t[:4]) for t in terms], axis=1)
    W = np.broadcast_to(np.array([t[4] for t in terms]) * h ** 2, X.shape)
    exact = (W * X).sum(1) * factor
    lib = out[nv:].reshape((n + 1,) * 3)[1:-1, 1:-1, 1:-1].ravel() - exact
    plain = f32(plain_sum(W, X) * f32(factor)) - exact
    print(f"{disc} {path}: {rms(lib) / rms(exact):.3e}, one chain {rms(plain) / rms(exact):.3e}, "
          f"ratio {rms(lib) / rms(plain):.3f}")
    assert rms(lib) <= rms(plain)


@pytest.mark.parametrize("disc,box,L", [("P1P1", (3, 1, 2), 3), ("P1P1", (5, 1, 1), 3), ("P2P1", (3, 1, 2), 3),
                                        ("P2P1", (1, 1, 5), 3)])
def test_no_common_factor(disc, box, L):
    """Mesh widths that are no power of two: no error of the factor that scales a
    row.  With integers as input the terms of these rows are integers times a unit
    of the row and add up exactly, so that a row is its sum times a factor, rounded
    once: half a unit in the last place, and a hundredth of it for the factor (in
    two parts: 2^-46).  A factor rounded to FP32 is off by up to as much again, and
    all rows with it."""
    from paper_2010_13513_gb300 import hhg
    lc = 0 if disc == "P1P1" else 1
    pb = lib_problem(box, L, disc, lc=lc, solve="mixed")
    lev = oracle_hierarchy(box, L, disc, lc=lc).lv[L]
    x = np.random.default_rng(5).integers(1, 1000, size=lev.size).astype(np.float64)
    x[:3 * lev.nv] *= np.tile(lev.vint, 3)
    inner = np.concatenate([lev.vint] * 3)
    u, p = lev.split(x)
    only_u, only_p = lev.join(u, 0 * p), lev.join([0 * c for c in u], p)

    def check(name, out, exact):
        s = np.abs(exact) > 1e-6 * np.abs(exact).max()               # (exact zeros are not, in the oracle)
        e = np.abs(out[s] - exact[s]) / np.spacing(np.abs(exact[s]).astype(F))
        print(f"{disc} {box} {name}: {e.max():.3f} units in the last place, {s.sum()} rows")
        assert s.sum() > 1000 and e.max() <= 0.51

    y = pb.new_vector(L, hhg.FP32)
    pb.apply(L, "BT", pb.to_device(L, only_p, hhg.FP32), y)
    check("B^T p", pb.to_host(L, y)[:3 * lev.nv][inner],
          np.concatenate([(lev.B[c].T @ p) * lev.vint for c in range(3)])[inner])
    if disc == "P1P1":
        pb.apply(L, "FULL", pb.to_device(L, only_u, hhg.FP32), y)
        check("full operator", pb.to_host(L, y)[:3 * lev.nv][inner], np.concatenate([lev.A @ c for c in u])[inner])
    # the vertex colour that a sweep updates first: - (the rest of the row) / diagonal
    first = lev.phases[0]
    exact = np.concatenate([(lev.Adiag * c - lev.A @ c)[first] / lev.Adiag[first] for c in u])
    # (the resident smoother of P2-P1 rounds the edge terms' sum on the way)
    for ctas in (0, 4) if disc == "P1P1" else (0,):
        pb.set_level_smoother(L, ctas, prec=hhg.FP32)
        xd = pb.to_device(L, only_u, hhg.FP32)
        pb.smooth(L, hhg.Params.make(1, 1, 0, 1, "f", 1, OMEGA_INV[disc]), 1, xd, pb.new_vector(L, hhg.FP32))
        out = lev.split(pb.to_host(L, xd))[0]
        check(f"first colour, {ctas} CTAs", np.concatenate([c[first] for c in out]), exact)
