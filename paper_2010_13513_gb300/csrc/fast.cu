// Gauss-Seidel phases of the inexact Uzawa velocity step as separate launches.
//
// The term count of every row is a compile-time constant (generated at build
// time from the stencil builder, structure.inc), so each row is one fully
// unrolled sequence of independent loads and FMAs.  The weights and the
// linear offsets of the level (array * array_stride + di + dj*sx + dk*sy) are
// __grid_constant__ kernel parameters: every term reads its weight and offset
// from the constant bank, not from memory.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "batch.h"
#include "fast.h"
#include "kernels.h"
#include "structure.inc"

namespace hhg {
namespace {

__device__ __forceinline__ int64_t fsite(const Geo& g, int i, int j, int k) {
  return int64_t(i + 1) + int64_t(j + 1) * g.sx + int64_t(k + 1) * g.sy;
}

// Programmatic dependent launch (Gauss-Seidel phases): a kernel launched with
// the programmatic-serialization attribute may start while its predecessor in
// the stream finishes; it waits here until the predecessor has completed and
// its writes are visible (no-op for an ordinary launch), and each block
// signals its own successor once its work is done.  (In the stencil-row
// kernels the wait doubles the register count of the 25-way row dispatch, so
// those launch plainly.)
__device__ __forceinline__ void pdl_wait() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void pdl_trigger() { cudaTriggerProgrammaticLaunchCompletion(); }

// the work item's table (a device copy) staged in the block's shared memory,
// so that the unrolled terms read their weights and offsets from there
template <class Tab>
__device__ __forceinline__ const Tab& stage_table(const Tab* src) {
  extern __shared__ __align__(16) unsigned char kb_tab_smem[];
  static_assert(sizeof(Tab) % 4 == 0, "tables are copied as 4-byte words");
  const unsigned* s = reinterpret_cast<const unsigned*>(src);
  unsigned* d = reinterpret_cast<unsigned*>(kb_tab_smem);
  for (int q = threadIdx.x; q < int(sizeof(Tab) / 4); q += blockDim.x) d[q] = __ldg(s + q);
  __syncthreads();
  return *reinterpret_cast<const Tab*>(kb_tab_smem);
}

// -------------------------------------------------- Gauss-Seidel phase kernel
// sum over the 2^LP lanes of a group of consecutive lanes (all lanes of the
// warp take part)
template <int LP, class T>
__device__ __forceinline__ T lane_sum(T v) {
#pragma unroll
  for (int m = (1 << LP) >> 1; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// grid: x over the (i', j) plane (i' = i, or i / 4 for a vertex colour) times
// 2^LP lanes per site, z = k.  With LP > 0 the lanes of a site take every
// 2^LP-th term and add their sums by shuffles: shorter dependent chains and
// more threads for the small levels, whose phases are latency-bound.
// NC = 3: the three velocity components at once (u, rhs: block vectors);
// NC = 1: one component (u, rhs point to that component's first group array)
template <int DISC, int VARNU, int GRP, class T, int LP, int NC, int T0, int N1, class Tab>
__device__ __forceinline__ void gs_site(const uint3 bid, const Geo& g, T* __restrict__ u, const T* __restrict__ rhs,
                                        T inv_diag, int colour, const Tab& tab) {
  constexpr int ox = GRP == 1 || GRP == 4 || GRP == 5 || GRP == 7;
  constexpr int oy = GRP == 2 || GRP == 4 || GRP == 6 || GRP == 7;
  constexpr int oz = GRP == 3 || GRP == 5 || GRP == 6 || GRP == 7;
  constexpr int P = 1 << LP;
  const int k = bid.z;
  const int w = colour >= 0 ? (g.nx + 1 + 3) / 4 : g.nx + 1 - ox;
  const int q = bid.x * blockDim.x + threadIdx.x;
  const int site = q >> LP, p = q & (P - 1);
  const int j = site / w;
  int i = site - j * w;
  if (colour >= 0) i = 4 * i + (((colour - j - k) % 4) + 4) % 4;
  const int Px = 2 * i + ox, Py = 2 * j + oy, Pz = 2 * k + oz;
  const bool ok = Px > 0 && Py > 0 && Pz > 0 && Px < 2 * g.nx && Py < 2 * g.ny && Pz < 2 * g.nz;
  if (LP == 0 && !ok) return;
  const int64_t idx = ok ? fsite(g, i, j, k) : 0;
  const int64_t cs = int64_t(g.G) * g.arr;
  const T* us = u + idx;
  T a0 = T(0), a1 = T(0), a2 = T(0);
  if constexpr (LP == 0) {
#pragma unroll
    for (int t = 1; t < N1; ++t) {             // the diagonal is the first term
      const T wt = tab.w[T0 + t];
      const int o = tab.off[T0 + t];
      a0 += wt * us[o];
      if (NC == 3) {
        a1 += wt * us[o + cs];
        a2 += wt * us[o + 2 * cs];
      }
    }
  } else {
    if (ok) {
#pragma unroll
      for (int t0 = 1; t0 < N1; t0 += P) {
        const int t = t0 + p;
        if (t < N1) {
          const T wt = tab.w[T0 + t];
          const int o = tab.off[T0 + t];
          a0 += wt * us[o];
          if (NC == 3) {
            a1 += wt * us[o + cs];
            a2 += wt * us[o + 2 * cs];
          }
        }
      }
    }
    a0 = lane_sum<LP>(a0);                     // whole warps: the grid covers whole blocks
    if (NC == 3) {
      a1 = lane_sum<LP>(a1);
      a2 = lane_sum<LP>(a2);
    }
    if (!ok || p != 0) return;
  }
  T einv = T(1);
  if (VARNU) einv = T(g.eisc[k]);
  const int64_t o0 = int64_t(GRP) * g.arr + idx;
  u[o0] = (rhs[o0] * einv - a0) * inv_diag;
  if (NC == 3) {
    u[o0 + cs] = (rhs[o0 + cs] * einv - a1) * inv_diag;
    u[o0 + 2 * cs] = (rhs[o0 + 2 * cs] * einv - a2) * inv_diag;
  }
}

template <int DISC, int VARNU, int GRP, class T, int LP, int NC>
__global__ void __launch_bounds__(256)
    k_gs_fast(Geo g, T* __restrict__ u, const T* __restrict__ rhs, T inv_diag, int colour,
              const __grid_constant__ FastTab<T, gen::S<DISC, VARNU, OP_A>::N> tab) {
  using S = gen::S<DISC, VARNU, OP_A>;
  constexpr gen::RowS rw = S::rows[GRP];       // component-0 row of the group; all terms in segment 1
  static_assert(rw.n0 == 0 && rw.n2 == 0, "A rows carry only nu-scaled terms");
  pdl_wait();
  gs_site<DISC, VARNU, GRP, T, LP, NC, rw.t0, rw.n1>(blockIdx, g, u, rhs, inv_diag, colour, tab);
  pdl_trigger();
}
template <class T, class Tab>
struct GsA { Geo g; T* u; const T* rhs; T inv_diag; int colour; const Tab* tab; };
template <int DISC, int VARNU, int GRP, class T, int LP, int NC>
__global__ void __launch_bounds__(256) kb_gs_fast(const void* items, int n) {
  using S = gen::S<DISC, VARNU, OP_A>;
  using Tab = FastTab<T, S::N>;
  constexpr gen::RowS rw = S::rows[GRP];
  uint3 bid, gd;
  const auto& it = batch_item<GsA<T, Tab>>(items, n, bid, gd);
  const GsA<T, Tab>& a = it.a;
  const Tab& tab = stage_table(a.tab);
  gs_site<DISC, VARNU, GRP, T, LP, NC, rw.t0, rw.n1>(bid, a.g, a.u, a.rhs, a.inv_diag, a.colour, tab);
}

}  // namespace

// ================================================================= launchers
// Launches of at most about one wave (152 SMs x 8 blocks) may overlap their
// predecessor's tail (programmatic dependent launch): there the launch gap is
// a large part of the kernel time.  Longer grids are launched plainly.
constexpr int64_t kPdlMaxBlocks = 152 * 8;

template <class K, class... A>
void launch_pdl(K kernel, dim3 grd, dim3 blk, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grd;
  cfg.blockDim = blk;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = int64_t(grd.x) * grd.y * grd.z <= kPdlMaxBlocks ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

// launch geometry of a Gauss-Seidel phase
struct GsGeo {
  dim3 grd, blk;
  int lp;            // log2 of the lanes per site
};
inline GsGeo gs_geo(const Geo& g, int grp, int colour, const Shape& sh) {
  const int nt = grp == 0 && sh.gs_threads0 ? sh.gs_threads0 : sh.gs_threads;
  const int nl = grp == 0 ? sh.gs_lanes0 : sh.gs_lanes;
  GsGeo r;
  r.lp = nl == 4 ? 2 : nl == 2 ? 1 : 0;
  r.blk = dim3(nt, 1, 1);
  const int ni = colour >= 0 ? (g.nx + 1 + 3) / 4 : g.nx + 1;
  const int64_t plane = int64_t(ni) * (g.ny + 1) << r.lp;
  r.grd = dim3(unsigned((plane + nt - 1) / nt), 1, g.nz + 1);
  return r;
}

// the group and lane count of a phase as compile-time constants
template <class F>
void by_group_lanes(int grp, int lp, F&& f) {
  auto by_lanes = [&](auto gc) {
    if (lp == 2) f(gc, std::integral_constant<int, 2>{});
    else if (lp == 1) f(gc, std::integral_constant<int, 1>{});
    else f(gc, std::integral_constant<int, 0>{});
  };
  switch (grp) {
    case 0: by_lanes(std::integral_constant<int, 0>{}); break;
    case 1: by_lanes(std::integral_constant<int, 1>{}); break;
    case 2: by_lanes(std::integral_constant<int, 2>{}); break;
    case 3: by_lanes(std::integral_constant<int, 3>{}); break;
    case 4: by_lanes(std::integral_constant<int, 4>{}); break;
    case 5: by_lanes(std::integral_constant<int, 5>{}); break;
    case 6: by_lanes(std::integral_constant<int, 6>{}); break;
    case 7: by_lanes(std::integral_constant<int, 7>{}); break;
    default: break;
  }
}

#if defined(HHG_FAST_BATCHED)
// ------------------------------------------------ batch recording (kb_*)
template <int DISC, int VARNU, class T>
void record_gs(const Geo& g, const void* tab, int grp, int colour, double inv_diag, T* u, const T* rhs,
               const Shape& sh, int comp) {
  using Tab = FastTab<T, gen::S<DISC, VARNU, OP_A>::N>;
  const GsGeo gg = gs_geo(g, grp, colour, sh);
  const Tab* dtab = static_cast<const Tab*>(g_rec->table(tab, sizeof(Tab)));
  const int64_t cs = comp < 0 ? 0 : int64_t(comp) * g.G * g.arr;   // the component's first group array
  by_group_lanes(grp, gg.lp, [&](auto gc, auto lc) {
    constexpr int GRP = decltype(gc)::value, LP = decltype(lc)::value;
    if constexpr (DISC == 2 || GRP == 0) {
      const void* fn = comp < 0 ? reinterpret_cast<const void*>(kb_gs_fast<DISC, VARNU, GRP, T, LP, 3>)
                                : reinterpret_cast<const void*>(kb_gs_fast<DISC, VARNU, GRP, T, LP, 1>);
      g_rec->add(fn, gg.grd, gg.blk, sizeof(Tab), 1, GsA<T, Tab>{g, u + cs, rhs + cs, T(inv_diag), colour, dtab});
    }
  });
}
#else
// ------------------------------------------------------- plain launches
template <int DISC, int VARNU, class T>
void launch_gs_fast(const Geo& g, const void* tab, int grp, int colour, double inv_diag, T* u, const T* rhs,
                    const Shape& sh, int comp, cudaStream_t s) {
  using Tab = FastTab<T, gen::S<DISC, VARNU, OP_A>::N>;
  const Tab& tb = *static_cast<const Tab*>(tab);
  const GsGeo gg = gs_geo(g, grp, colour, sh);
  ++g_launches;
  const int64_t cs = comp < 0 ? 0 : int64_t(comp) * g.G * g.arr;   // the component's first group array
  by_group_lanes(grp, gg.lp, [&](auto gc, auto lc) {
    constexpr int GRP = decltype(gc)::value, LP = decltype(lc)::value;
    if constexpr (DISC == 2 || GRP == 0) {
      if (comp < 0)
        launch_pdl(k_gs_fast<DISC, VARNU, GRP, T, LP, 3>, gg.grd, gg.blk, s, g, u, rhs, T(inv_diag), colour, tb);
      else
        launch_pdl(k_gs_fast<DISC, VARNU, GRP, T, LP, 1>, gg.grd, gg.blk, s, g, u + cs, rhs + cs, T(inv_diag),
                   colour, tb);
    }
  });
}
#endif

#if (!defined(HHG_FAST_ONLY) || HHG_FAST_ONLY == 64) && !defined(HHG_FAST_BATCHED)
int fast_terms(int disc, int varnu, int op) {
#define HHG_N(D, V, O) if (disc == D && varnu == V && op == O) return gen::S<D, V, O>::N;
  HHG_N(1, 0, OP_FULL) HHG_N(1, 0, OP_A) HHG_N(1, 0, OP_BT) HHG_N(1, 0, OP_BC)
  HHG_N(1, 1, OP_FULL) HHG_N(1, 1, OP_A) HHG_N(1, 1, OP_BT) HHG_N(1, 1, OP_BC)
  HHG_N(2, 0, OP_FULL) HHG_N(2, 0, OP_A) HHG_N(2, 0, OP_BT) HHG_N(2, 0, OP_BC)
  HHG_N(2, 1, OP_FULL) HHG_N(2, 1, OP_A) HHG_N(2, 1, OP_BT) HHG_N(2, 1, OP_BC)
#undef HHG_N
  return -1;
}

#endif

#if defined(HHG_FAST_BATCHED)
// run-time dispatch over (disc, varnu, op) of the recorders
template <class T>
void fast_gs_record(int disc, int varnu, const Geo& g, const void* tab, int grp, int colour, double inv_diag, T* u,
                    const T* rhs, const Shape& sh, int comp) {
  if (disc == 1 && !varnu) record_gs<1, 0, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp);
  else if (disc == 1) record_gs<1, 1, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp);
  else if (!varnu) record_gs<2, 0, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp);
  else record_gs<2, 1, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp);
}

#if HHG_FAST_ONLY == 64
template void fast_gs_record<double>(int, int, const Geo&, const void*, int, int, double, double*, const double*,
                                     const Shape&, int);
#else
template void fast_gs_record<float>(int, int, const Geo&, const void*, int, int, double, float*, const float*,
                                    const Shape&, int);
#endif
#else
// run-time dispatch over (disc, varnu, op); while a batch records, the
// recorders (the batched translation units) take the launch
template <class T>
void fast_gs(int disc, int varnu, const Geo& g, const void* tab, int grp, int colour, double inv_diag, T* u,
             const T* rhs, const Shape& sh, cudaStream_t s, int comp) {
  if (g_rec) return fast_gs_record<T>(disc, varnu, g, tab, grp, colour, inv_diag, u, rhs, sh, comp);
  if (disc == 1 && !varnu) launch_gs_fast<1, 0, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp, s);
  else if (disc == 1) launch_gs_fast<1, 1, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp, s);
  else if (!varnu) launch_gs_fast<2, 0, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp, s);
  else launch_gs_fast<2, 1, T>(g, tab, grp, colour, inv_diag, u, rhs, sh, comp, s);
}

// HHG_FAST_ONLY = 64 / 32 compiles one precision (the build compiles this
// file once per precision, in parallel)
#if !defined(HHG_FAST_ONLY) || HHG_FAST_ONLY == 64
template void fast_gs<double>(int, int, const Geo&, const void*, int, int, double, double*, const double*, const Shape&,
                              cudaStream_t, int);
#endif
#if !defined(HHG_FAST_ONLY) || HHG_FAST_ONLY == 32
template void fast_gs<float>(int, int, const Geo&, const void*, int, int, double, float*, const float*, const Shape&,
                             cudaStream_t, int);
#endif
#endif

}  // namespace hhg
