// Shared-memory-resident inexact Uzawa smoother for small levels (small.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace hhg {

// scalar arguments of one smoother launch
struct SmallArgs {
  int iterations;          // Uzawa iterations
  int xi;                  // Gauss-Seidel sweeps per velocity step
  int ahat;                // HHG_AHAT_F / HHG_AHAT_S
  double inv_omega_inv;    // omega = 1 / omega^{-1}
  double inv_diag[8];      // 1 / diag(A) per group
};

constexpr int kResMaxTerms = 640;   // component-0 rows of A, the rows of B^T, the row of (B, -C)
constexpr int kResMaxC = 15;        // lattice offsets of the C stencil

// run-time weights of one level: the rows of A of component 0, of B^T and of
// (B, -C) in the order of the generated structure (the smoother reads them with a
// variable viscosity only, the full operator's rows (rows.cu) the interior C
// terms of P1-P1 with a constant one too), and the C stencil of the pressure row clipped to the
// domain per boundary class (27 x the stencil's offsets, class
// ci + 3 cj + 9 ck with c = 0 on the low face, 1 inside, 2 on the high face)
template <class T>
struct ResTabs {
  T w[kResMaxTerms];
  T wc[27 * kResMaxC];
};

constexpr int kResidentThreads = 1024;            // most threads per CTA (128..1024, a multiple of 32)
constexpr int kResidentMaxCtas = 16;              // largest (non-portable) cluster
constexpr size_t kResidentSmemMax = 225 * 1024;   // dynamic shared memory per CTA (static use below 2 KB)

// shared memory per CTA (bytes) of a cluster of `ctas` CTAs on the level: CTA
// c owns the k planes [c (nz+1) / C, (c+1) (nz+1) / C) of every array and
// keeps them, with one halo plane below and above, next to its right-hand
// sides and site tables (a compact layout without the tables where that does
// not fit: resident_compact)
bool resident_compact(int disc, int varnu, const Geo& g, int ctas, int prec);
size_t resident_smem(int disc, int varnu, const Geo& g, int ctas, int prec);
// true if `ctas` CTAs can hold the level (every CTA owns a plane, the slab
// fits the shared memory, the cluster can be scheduled).  Sets the kernel's
// shared-memory and cluster-size attributes; call before any launch with
// this CTA count and outside stream capture.
bool resident_feasible(int disc, int varnu, int prec, const Geo& g, int ctas);

// `iterations` inexact Uzawa iterations of a level in one launch of a
// cluster of `ctas` CTAs of `threads` threads; `tabs`: device table of the
// level.  Returns 0 or -1 (launch failure).
template <class T>
int uzawa_resident(int disc, int varnu, const Geo& g, int ctas, int threads, T* x, const T* b, const double* inv_ml,
                   const SmallArgs& a, const ResTabs<T>* tabs, cudaStream_t s);

}  // namespace hhg
