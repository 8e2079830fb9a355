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
