// Multicolour Gauss-Seidel phases of the inexact Uzawa velocity step (Sec.
// 3.2) as separate launches, for the levels that do not fit the
// shared-memory-resident smoother.
//
// A thread updates one site of one component (P1-P1: of all three, which share
// the index arithmetic: a sweep with constant viscosity at 2.1 million sites 55
// us with a component per thread, 34 us).  The row is unrolled from the
// generated structure; with a constant viscosity its weights are immediates
// (the sum scaled by the inverse diagonal: weights.h), with a variable one the
// group's row is a kernel parameter.  Offsets are formed from the array stride
// and the pitches, uniform for the launch, and added to a 32-bit site index, so
// that a term is little more than its load and its FMA.  (The kernels these
// replace passed weights and linear offsets of all groups as a 4.5 KB
// parameter table, one thread or up to four lanes per site for all three
// components, about six instructions per term.)
//
// A vertex row of P2-P1 reads 44 edge DoFs that no vertex phase changes.
// gs_vertex_phases sums these terms once for all four colours, with
// consecutive sites in consecutive lanes; a launch per colour, whose lanes lie
// four sites apart (four times the sectors per access), then reads the six
// vertex neighbours only.  One smoothing step (three sweeps, FP32) with full rows on
// all components / component by component / on shared edge sums: level 6 211 / 324
// / 213 us, 1.1 million sites (2x2x1 cubes) 894 / 842 / 796 us, level 7 1,725 /
// 1,577 / 1,503 us; with variable viscosity at 1.1 million 1,019 / 1,001 / 963 us.
//
// Bound: launch latency on level 5, L1/L2 loads on level 6, HBM on level 7 (an
// edge phase reads the whole velocity, 217 MB in FP32).  Measured, one forward
// sweep of P2-P1: FP32 level 5 / 6 / 7 28.8 / 59.5 / 543 us before, 23.8 / 59.9
// / 439 us now (level 7 with the shared edge sums); FP64 level 4 44 us before,
// 31 us; P1-P1 at 2.1 / 17 million sites, constant viscosity, 47.7 / 378 us
// before, 34.1 / 368 us, variable viscosity 64.9 / 443 us before, 53.4 / 426 us.
// Programmatic launches pay at every size: limited to one wave of
// blocks, the level-6 sweep takes 78 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "at.h"
#include "batch.h"
#include "gs.h"
#include "kernels.h"
#include "structure.inc"
#include "weights.h"

namespace hhg {
namespace {

enum { kAllTerms = 0, kVertexTerms = 1, kEdgeTerms = 2 };

template <class T, int NW>
struct GsA { Geo g; T* u; const T* rhs; T inv_diag; int colour, comp; T w[NW]; };
template <int DISC, int VARNU, int GRP>
constexpr int row_nw() { return VARNU ? gen::S<DISC, VARNU, OP_A>::rows[GRP].n1 : 1; }

// the terms of row GRP behind the diagonal that pass the filter, at the site
// of 32-bit index i; w: the row's weights (NW = 1: immediates, weights.h)
template <int DISC, class S, int GRP, int SEL, int NW, class T, int... I>
__device__ __forceinline__ T row_sum(const Geo& g, const T* u, const Lines<T>& at, const T (&w)[NW],
                                     std::integer_sequence<int, I...>) {
  T a[3] = {};
  ([&] {
    constexpr int e = S::rows[GRP].t0 + 1 + I;     // the diagonal is the first term
    constexpr gen::OffT o = S::off[e];
    if constexpr (SEL == kAllTerms || (SEL == kVertexTerms) == (o.arr == 0)) {
      T wt;
      if constexpr (NW > 1) {
        wt = w[1 + I];
      } else {
        constexpr double r = row_weight<S, e, T>(kScaleA<DISC>);
        wt = T(r);
      }
      a[I % 3] = fma(wt, at.template get<o.di, o.dj, o.dk>(u + o.arr * g.arr), a[I % 3]);
    }
  }(), ...);
  return (a[0] + a[1]) + a[2];
}
// (r - s) / diagonal: a row's new value from its right-hand side and its other
// terms.  Constant viscosity: s in the scale of the row's weights, and with
// vertex terms only r comes divided (edge_sums)
template <int DISC, int VARNU, int GRP, int SEL, class T>
__device__ __forceinline__ T new_value(T r, T s, T inv_diag) {
  if constexpr (VARNU != 0) {
    return (r - s) * inv_diag;
  } else {
    using S = gen::S<DISC, VARNU, OP_A>;
    constexpr gen::RowS rw = S::rows[GRP];
    static_assert(int_weights<S>(rw.t0, rw.n1, kScaleA<DISC>), "the scaled weights are small integers");
    constexpr Factor<T> f = make_factor<T>(1.0 / row_weight<S, rw.t0, T>(kScaleA<DISC>));
    return minus_scaled(SEL == kVertexTerms ? r : r * inv_diag, f, s);
  }
}

// Programmatic dependent launch: a phase may start while its predecessor in
// the stream finishes; it waits here until the predecessor's writes are
// visible (no-op for an ordinary launch) and signals its own successor once
// its work is done.
__device__ __forceinline__ void pdl_wait() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void pdl_trigger() { cudaTriggerProgrammaticLaunchCompletion(); }

// grid: x over the sites of the (i, j) plane (a vertex colour: quads of four
// sites of a row), y = component (NC = 3: a thread takes all three), z = plane
template <int DISC, int VARNU, int GRP, int SEL, int NC, class T, int NW>
__device__ __forceinline__ void gs_site(const uint3 bid, const GsA<T, NW>& a) {
  using S = gen::S<DISC, VARNU, OP_A>;
  constexpr gen::RowS rw = S::rows[GRP];
  static_assert(rw.n0 == 0 && rw.n2 == 0 && rw.n1 <= kGsTerms, "A rows carry only nu-scaled terms");
  constexpr int G = DISC == 2 ? 8 : 1;
  constexpr int ox = (0xB2 >> GRP) & 1, oy = (0xD4 >> GRP) & 1, oz = (0xE8 >> GRP) & 1;
  const Geo& g = a.g;
  const int k = int(bid.z) + (oz ? 0 : 1);         // planes with interior DoFs
  const int w = GRP == 0 ? (g.nx + 3) / 4 : g.nx, q = bid.x * blockDim.x + threadIdx.x;
  const int jj = q / w, j = jj + (oy ? 0 : 1);
  int i = q - jj * w;
  if (GRP == 0) i = 4 * i + ((a.colour - j - k) & 3);
  if (j >= g.ny || i >= g.nx || (!ox && i == 0)) return;
  const int kb = kByPlane<DISC, T> ? k : 0;          // the plane that offsets count from
  const Lines<T> at(g, unsigned(i + 1) + unsigned(j + 1) * unsigned(g.sx) + unsigned(k - kb + 1) * unsigned(g.sy));
  const int64_t base = int64_t(a.comp + int(bid.y)) * G * g.arr;
  T* u = a.u + base;
  const T* rhs = a.rhs + (SEL == kVertexTerms ? int64_t(bid.y) * g.arr : base + GRP * g.arr);
  if constexpr (kByPlane<DISC, T>) {
    u += kb * g.sy;
    rhs += kb * g.sy;
  }
  if constexpr (NC == 1) {
    T r = ld_at(rhs, at.site());
    const T s = row_sum<DISC, S, GRP, SEL>(g, u, at, a.w, std::make_integer_sequence<int, rw.n1 - 1>{});
    if (VARNU && SEL != kVertexTerms) r *= T(g.eisc[k]);
    ref_at(u + GRP * g.arr, at.site()) = new_value<DISC, VARNU, GRP, SEL>(r, s, a.inv_diag);
  } else {
    static_assert(DISC == 1 && SEL == kAllTerms && GRP == 0, "one array per component");
    T v[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int64_t bc = int64_t(a.comp + int(bid.y) + c) * G * g.arr;
      T r = ld_at(a.rhs + kb * g.sy + bc + GRP * g.arr, at.site());
      const T s = row_sum<DISC, S, GRP, SEL>(g, a.u + bc + kb * g.sy, at, a.w, std::make_integer_sequence<int, rw.n1 - 1>{});
      if (VARNU) r *= T(g.eisc[k]);
      v[c] = new_value<DISC, VARNU, GRP, SEL>(r, s, a.inv_diag);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
      ref_at(a.u + int64_t(a.comp + int(bid.y) + c) * G * g.arr + kb * g.sy + GRP * g.arr, at.site()) = v[c];
  }
}
template <int DISC, int VARNU, int GRP, int SEL, int NC, class T>
__global__ void __launch_bounds__(256) k_gs(const __grid_constant__ GsA<T, row_nw<DISC, VARNU, GRP>()> a) {
  pdl_wait();
  gs_site<DISC, VARNU, GRP, SEL, NC>(blockIdx, a);
  pdl_trigger();
}
template <int DISC, int VARNU, int GRP, int SEL, int NC, class T>
__global__ void __launch_bounds__(256) kb_gs(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<GsA<T, row_nw<DISC, VARNU, GRP>()>>(items, n, bid, gd);
  gs_site<DISC, VARNU, GRP, SEL, NC>(bid, it.a);
}

// t = rhs - (edge terms of the vertex row) at the interior vertices (constant
// viscosity: divided by the diagonal, the scale of u); block: 32 x 8 sites of the
// plane, a few planes per block on levels that fill the GPU (their lines then
// meet in L1)
template <class T, int NW>
struct EdgeA { Geo g; const T* u; const T* rhs; T* t; T inv_diag; int kp; T w[NW]; };
template <int VARNU, class T, int NW>
__device__ __forceinline__ void edge_sums(const uint3 bid, const EdgeA<T, NW>& a) {
  using S = gen::S<2, VARNU, OP_A>;
  const Geo& g = a.g;
  const int comp = int(bid.z) % 3, k0 = 1 + int(bid.z) / 3 * a.kp;
  const int i = 1 + bid.x * 32 + int(threadIdx.x & 31), j = 1 + bid.y * 8 + int(threadIdx.x >> 5);
  if (i >= g.nx || j >= g.ny) return;
  const T* u = a.u + int64_t(comp) * 8 * g.arr;
  const T* rhs = a.rhs + int64_t(comp) * 8 * g.arr;
  T* t = a.t + int64_t(comp) * g.arr;
#pragma unroll 1
  for (int k = k0; k < min(k0 + a.kp, g.nz); ++k) {
    const Lines<T> at(g, unsigned(i + 1) + unsigned(j + 1) * unsigned(g.sx) + unsigned(k + 1) * unsigned(g.sy));
    const T s = row_sum<2, S, 0, kEdgeTerms>(g, u, at, a.w, std::make_integer_sequence<int, S::rows[0].n1 - 1>{});
    T r = ld_at(rhs, at.site());
    if (VARNU) r *= T(g.eisc[k]);
    ref_at(t, at.site()) = VARNU ? r - s : new_value<2, VARNU, 0, kEdgeTerms>(r, s, a.inv_diag);
  }
}
template <int VARNU, class T>
__global__ void __launch_bounds__(256) k_edge_sums(const __grid_constant__ EdgeA<T, row_nw<2, VARNU, 0>()> a) {
  edge_sums<VARNU>(blockIdx, a);
}
template <int VARNU, class T>
__global__ void __launch_bounds__(256) kb_edge_sums(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<EdgeA<T, row_nw<2, VARNU, 0>()>>(items, n, bid, gd);
  edge_sums<VARNU>(bid, it.a);
}

template <class A>
void launch(const void* kernel, const void* batched, dim3 grd, int threads, bool pdl, const A& a, cudaStream_t s) {
  if (g_rec) return g_rec->add(batched, grd, dim3(threads), 0, 1, a);
  ++g_launches;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grd;
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  void* args[] = {const_cast<A*>(&a)};
  cudaLaunchKernelExC(&cfg, kernel, args);
}

template <int DISC, int VARNU, int GRP, int SEL, class T>
void launch_phase(const Geo& g, const GsRows<T>& rows, int colour, T* u, const T* rhs, int comp, int ncomp, int threads,
                  cudaStream_t s) {
  constexpr int NW = row_nw<DISC, VARNU, GRP>();
  constexpr int oy = (0xD4 >> GRP) & 1, oz = (0xE8 >> GRP) & 1;
  GsA<T, NW> a{g, u, rhs, rows.inv_diag[GRP], colour, comp, {}};
  if (NW > 1) std::copy(rows.w[GRP], rows.w[GRP] + NW, a.w);
  // j from 1 (or 0, odd groups) to ny - 1, k the same
  const int w = GRP == 0 ? (g.nx + 3) / 4 : g.nx, nj = g.ny - (oy ? 0 : 1), nk = g.nz - (oz ? 0 : 1);
  if (nj < 1 || nk < 1) return;
  // P1-P1: a thread takes the three components of a site
  constexpr int NC = DISC == 1 ? 3 : 1;
  const dim3 grd(unsigned((w * nj + threads - 1) / threads), ncomp, nk);
  if (NC == 3 && ncomp == 3)
    return launch(reinterpret_cast<const void*>(k_gs<DISC, VARNU, GRP, SEL, NC, T>),
                  reinterpret_cast<const void*>(kb_gs<DISC, VARNU, GRP, SEL, NC, T>), dim3(grd.x, 1, nk), threads, true,
                  a, s);
  launch(reinterpret_cast<const void*>(k_gs<DISC, VARNU, GRP, SEL, 1, T>),
         reinterpret_cast<const void*>(kb_gs<DISC, VARNU, GRP, SEL, 1, T>), grd, threads, true, a, s);
}

template <int VARNU, class T>
void launch_vertex(const Geo& g, const GsRows<T>& rows, bool reverse, T* u, const T* rhs, T* t, int threads,
                   cudaStream_t s) {
  constexpr int NW = row_nw<2, VARNU, 0>();
  const int kp = int64_t(g.nx + 1) * (g.ny + 1) * (g.nz + 1) > 1000000 ? 4 : 1;
  EdgeA<T, NW> a{g, u, rhs, t, rows.inv_diag[0], kp, {}};
  if (NW > 1) std::copy(rows.w[0], rows.w[0] + NW, a.w);
  if (g.nx < 2 || g.ny < 2 || g.nz < 2) return;    // no interior vertex
  const dim3 grd((g.nx - 1 + 31) / 32, (g.ny - 1 + 7) / 8, 3 * ((g.nz - 1 + kp - 1) / kp));
  launch(reinterpret_cast<const void*>(k_edge_sums<VARNU, T>), reinterpret_cast<const void*>(kb_edge_sums<VARNU, T>),
         grd, 256, false, a, s);
  for (int c = 0; c < 4; ++c)
    launch_phase<2, VARNU, 0, kVertexTerms, T>(g, rows, reverse ? 3 - c : c, u, t, 0, 3, threads, s);
}

template <int VARNU, class T>
void phase_p2(const Geo& g, const GsRows<T>& rows, int grp, int colour, T* u, const T* rhs, int comp, int ncomp,
              int threads, cudaStream_t s) {
#define HHG_P(GRP) \
  case GRP: launch_phase<2, VARNU, GRP, kAllTerms, T>(g, rows, colour, u, rhs, comp, ncomp, threads, s); break;
  switch (grp) { HHG_P(0) HHG_P(1) HHG_P(2) HHG_P(3) HHG_P(4) HHG_P(5) HHG_P(6) HHG_P(7) default: break; }
#undef HHG_P
}

}  // namespace

template <class T>
void gs_phase(int disc, int varnu, const Geo& g, const GsRows<T>& rows, int grp, int colour, T* u, const T* rhs,
              int comp, int ncomp, int threads, cudaStream_t s) {
  if (disc == 2) {
    if (varnu) phase_p2<1, T>(g, rows, grp, colour, u, rhs, comp, ncomp, threads, s);
    else phase_p2<0, T>(g, rows, grp, colour, u, rhs, comp, ncomp, threads, s);
  } else if (varnu) {
    launch_phase<1, 1, 0, kAllTerms, T>(g, rows, colour, u, rhs, comp, ncomp, threads, s);
  } else {
    launch_phase<1, 0, 0, kAllTerms, T>(g, rows, colour, u, rhs, comp, ncomp, threads, s);
  }
}

template <class T>
void gs_vertex_phases(int varnu, const Geo& g, const GsRows<T>& rows, bool reverse, T* u, const T* rhs, T* t,
                      int threads, cudaStream_t s) {
  if (varnu) launch_vertex<1, T>(g, rows, reverse, u, rhs, t, threads, s);
  else launch_vertex<0, T>(g, rows, reverse, u, rhs, t, threads, s);
}

#define HHG_INST(T)                                                                                              \
  template void gs_phase<T>(int, int, const Geo&, const GsRows<T>&, int, int, T*, const T*, int, int, int,       \
                            cudaStream_t);                                                                       \
  template void gs_vertex_phases<T>(int, const Geo&, const GsRows<T>&, bool, T*, const T*, T*, int, cudaStream_t);
HHG_INST(double)
HHG_INST(float)

}  // namespace hhg
