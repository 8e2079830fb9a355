// The B^T rows and the pressure step of an inexact Uzawa iteration (Sec. 3.2,
// Eqs. uzawa-velocity / uzawa-pressure) on levels whose smoother runs as
// separate launches.
//
//  * k_bt: a thread owns a lattice cell and a component and evaluates all of
//    the component's rows there: the rows of the eight P2 groups read the same
//    15 pressure values, so these are loaded once, and the rest of the traffic
//    is the right-hand side in and tmp out, once each;
//  * k_pressure: the row of (B, -C) and the pressure update in one launch: a
//    thread owns a pressure site.  For P2-P1 the row reads no pressure and the
//    update is in place; the P1-P1 row does, so that the new pressures go to
//    the scratch vector and are copied back.
// All rows are unrolled from the generated structure; with a constant
// viscosity the weights are immediates (weights.h).  Boundary pressure
// rows keep the merged B terms (exact for inputs with zero Dirichlet
// velocities) and take the C stencil of their boundary class.
//
// Bound: HBM on the largest levels; below, the L1/L2 loads of the pressure
// row (156 for P2-P1), which is why a block of consecutive rows marches over
// a few planes: the lines of neighbouring rows and planes meet in L1.
// Measured, both rows and the update of one iteration against the three
// launches before: P2-P1 FP32 level 5 / 6 / 7: 24 / 49 / 236 us before, 12 / 31
// / 190 us now; P1-P1 with variable viscosity, 48 tetrahedra, level 6: 81 us
// before, 73 us (device times).  Larger P1-P1 levels in FP32 take four aligned
// sites per thread (quad.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "at.h"
#include "batch.h"
#include "kernels.h"
#include "quad.h"
#include "structure.inc"
#include "uzrows.h"
#include "weights.h"

namespace hhg {
namespace {

// 1 / the unit of the C terms of P1-P1
template <int VARNU>
constexpr double inv_unit_c() {
  if constexpr (VARNU) {
    return 1.0;
  } else {
    using S = gen::S<1, 0, OP_BC>;
    constexpr gen::RowS rw = S::rows[0];
    return 1.0 / c_unit<S>(rw.t0 + rw.n0, rw.n2);
  }
}

// weight of term E, of C (CT) or of B or B^T; constant viscosity (NW = 1): weights.h
template <int DISC, class S, int E, bool CT, class T, int NW>
__device__ __forceinline__ T rweight(const T (&w)[NW]) {
  if constexpr (NW > 1) {
    return w[E];
  } else {
    constexpr double K = CT ? inv_unit_c<0>() : kScaleB<DISC>, r = row_weight<S, E, T>(K);
    static_assert(int_weights<S>(E, 1, K), "the scaled weights are small integers");
    return T(r);
  }
}

// ------------------------------------------------------------------- B^T
template <class T, int NW>
struct BtA { Geo g; const T* x; const T* b; T* y; Factor<T> sb; T w[NW]; };   // b = null: y = B^T p; sb: h^2 / K
template <int DISC, int VARNU>
constexpr int bt_nw() { return VARNU ? gen::S<DISC, VARNU, OP_BT>::N : 1; }

template <int DISC, class S, int R, int NW, class T, int... I>
__device__ __forceinline__ T bt_row(const T (&p)[27], const T (&w)[NW], std::integer_sequence<int, I...>) {
  T a = T(0);
  ([&] {
    constexpr int e = S::rows[R].t0 + I;
    constexpr gen::OffT o = S::off[e];
    a = fma(rweight<DISC, S, e, false>(w), p[(o.di + 1) + 3 * (o.dj + 1) + 9 * (o.dk + 1)], a);
  }(), ...);
  return a;
}
// whether some row of B^T reads the pressure at offset q - 13 of the 27 neighbours
template <class S>
constexpr bool bt_reads(int q) {
  for (int e = 0; e < S::N; ++e)
    if ((S::off[e].di + 1) + 3 * (S::off[e].dj + 1) + 9 * (S::off[e].dk + 1) == q) return true;
  return false;
}
template <class S, class T, int... Q>
__device__ __forceinline__ void bt_load(const T* __restrict__ x, const Lines<T>& at, T (&p)[27],
                                        std::integer_sequence<int, Q...>) {
  ([&] {
    if constexpr (bt_reads<S>(Q)) p[Q] = at.template ld<Q % 3 - 1, Q / 3 % 3 - 1, Q / 9 - 1>(x);
  }(), ...);
}
template <int DISC, int VARNU, int R0, int NW, class T, int... GG>
__device__ __forceinline__ void bt_groups(const BtA<T, NW>& a, const T (&p)[27], unsigned at, int in,
                                        std::integer_sequence<int, GG...>) {
  using S = gen::S<DISC, VARNU, OP_BT>;
  const Geo& g = a.g;
  T bv[sizeof...(GG)];
  ((bv[GG] = a.b && (in >> GG & 1) ? ld_at(a.b + (R0 + GG) * g.arr, at) : T(0)), ...);
  ([&] {
    constexpr gen::RowS rw = S::rows[R0 + GG];
    static_assert(rw.n1 == 0 && rw.n2 == 0, "B^T is unscaled");
    const T v = bt_row<DISC, S, R0 + GG>(p, a.w, std::make_integer_sequence<int, rw.n0>{});
    if (in >> GG & 1) {
      T& y = ref_at(a.y + (R0 + GG) * g.arr, at);
      if constexpr (VARNU != 0) y = a.b ? bv[GG] - v : v;
      else y = a.b ? minus_scaled(bv[GG], a.sb, v) : scaled(a.sb, v);
    }
  }(), ...);
}

constexpr int kBtThreads = 128, kPressThreads = 256;

// grid x over the positions of the padded (i, j) plane, y = plane, z = component
template <int DISC, int VARNU, class T, int NW>
__device__ __forceinline__ void bt_body(const uint3 bid, const BtA<T, NW>& full) {
  constexpr int G = DISC == 2 ? 8 : 1;
  const Geo& g = full.g;
  const int q = bid.x * blockDim.x + threadIdx.x, j = q / g.sx, i = q - j * g.sx, k = bid.y;
  if (i >= g.nx || j >= g.ny) return;
  // groups with an interior DoF in the cell (order of kGroupOff)
  int in = 0;
#pragma unroll
  for (int gg = 0; gg < G; ++gg)
    if ((i > 0 || (0xB2 >> gg & 1)) && (j > 0 || (0xD4 >> gg & 1)) && (k > 0 || (0xE8 >> gg & 1))) in |= 1 << gg;
  const int kb = kByPlane<DISC, T> ? k : 0;          // the plane that offsets count from
  const Lines<T> at(g, unsigned(i + 1) + unsigned(j + 1) * unsigned(g.sx) + unsigned(k - kb + 1) * unsigned(g.sy));
  BtA<T, NW> a = full;
  a.x += kb * g.sy; a.y += kb * g.sy;
  if (a.b) a.b += kb * g.sy;
  T p[27];
  bt_load<gen::S<DISC, VARNU, OP_BT>>(a.x + 3 * G * g.arr, at, p, std::make_integer_sequence<int, 27>{});
  const auto groups = std::make_integer_sequence<int, G>{};
  if (DISC == 1) {                                 // the components share the pressures
    bt_groups<DISC, VARNU, 0>(a, p, at.site(), in, groups);
    bt_groups<DISC, VARNU, G>(a, p, at.site(), in, groups);
    bt_groups<DISC, VARNU, 2 * G>(a, p, at.site(), in, groups);
  } else if (bid.z == 0) {
    bt_groups<DISC, VARNU, 0>(a, p, at.site(), in, groups);
  } else if (bid.z == 1) {
    bt_groups<DISC, VARNU, G>(a, p, at.site(), in, groups);
  } else {
    bt_groups<DISC, VARNU, 2 * G>(a, p, at.site(), in, groups);
  }
}
template <int DISC, int VARNU, class T>
__global__ void __launch_bounds__(kBtThreads) k_bt(const __grid_constant__ BtA<T, bt_nw<DISC, VARNU>()> a) {
  bt_body<DISC, VARNU>(blockIdx, a);
}
template <int DISC, int VARNU, class T>
__global__ void __launch_bounds__(kBtThreads) kb_bt(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<BtA<T, bt_nw<DISC, VARNU>()>>(items, n, bid, gd);
  bt_body<DISC, VARNU>(bid, it.a);
}

// ---------------------------------------------------------- pressure step
template <class T, int NW>
struct PressA {
  Geo g; const T* x; const T* b; T* p; const double* inv_ml; double s; const ResTabs<T>* tabs; int kp;
  Factor<T> sb, sc;                                  // h^2 / K of B, h^3 times the unit of C
  T w[NW];
};
template <int DISC, int VARNU>
constexpr int bc_nw() { return VARNU ? gen::S<DISC, VARNU, OP_BC>::N : 1; }

// terms [T0, T0 + N) of the pressure row: three chains, one per component, the
// few C terms (whose diagonal stands in the middle) one chain
template <bool CT> constexpr int kChains = CT ? 1 : 3;
template <int DISC, class S, int T0, int N, bool CT, int NW, class T, int... J>
__device__ __forceinline__ T press_sum(const Geo& g, const T* __restrict__ x, const Lines<T>& at, const T (&w)[NW],
                                       std::integer_sequence<int, J...>) {
  constexpr int M = kChains<CT>;
  T a[3] = {};
  ([&] {
    constexpr int e = chain_term(J, N, M);
    if constexpr (e >= 0) {
      constexpr gen::OffT o = S::off[T0 + e];
      a[J % M] = fma(rweight<DISC, S, T0 + e, CT>(w), at.template ld<o.di, o.dj, o.dk>(x + o.arr * g.arr), a[J % M]);
    }
  }(), ...);
  return (a[0] + a[1]) + a[2];
}

// grid x over the positions of the padded (i, j) plane, y = groups of kp planes;
// ROW: the row itself into p, no update
template <int DISC, int VARNU, bool ROW, class T, int NW>
__device__ __forceinline__ void press_body(const uint3 bid, const PressA<T, NW>& a) {
  using S = gen::S<DISC, VARNU, OP_BC>;
  constexpr gen::RowS rw = S::rows[0];
  static_assert(rw.n1 == 0, "B is unscaled");
  constexpr int G = DISC == 2 ? 8 : 1;
  const Geo& g = a.g;
  const int q = bid.x * blockDim.x + threadIdx.x, j = q / g.sx, i = q - j * g.sx;
  if (i > g.nx || j > g.ny) return;
  const int k1 = min(int(bid.y + 1) * a.kp, g.nz + 1);
#pragma unroll 1
  for (int k = bid.y * a.kp; k < k1; ++k) {
    const int64_t idx = int64_t(i + 1) + int64_t(j + 1) * g.sx + int64_t(k + 1) * g.sy;
    const int kb = kByPlane<DISC, T> ? k : 0;        // the plane that offsets count from
    const Lines<T> at(g, unsigned(idx - kb * g.sy));
    T bv = T(0), ml = T(0);
    if constexpr (!ROW) {
      bv = __ldg(a.b + 3 * G * g.arr + idx);
      ml = T(a.s * __ldg(a.inv_ml + idx));
    }
    const T* x = a.x + idx;
    T v = press_sum<DISC, S, rw.t0, rw.n0, false>(g, a.x + kb * g.sy, at, a.w,
                                             std::make_integer_sequence<int, chain_steps(rw.n0, kChains<false>)>{});
    if (!VARNU) v = scaled(a.sb, v);
    if constexpr (rw.n2 > 0) {
      using SPT = gen::SP<DISC, VARNU, OP_BC>;
      T c;
      if (i == 0 || j == 0 || k == 0 || i == g.nx || j == g.ny || k == g.nz) {
        const int cls = (i == 0 ? 0 : i == g.nx ? 2 : 1) + 3 * (j == 0 ? 0 : j == g.ny ? 2 : 1) +
                        9 * (k == 0 ? 0 : k == g.nz ? 2 : 1);
        c = c_class<SPT>(g, x + 3 * G * g.arr, a.tabs->wc + cls * SPT::NCB, std::make_integer_sequence<int, SPT::NCB>{});
      } else {
        c = press_sum<DISC, S, rw.t0 + rw.n0, rw.n2, true>(g, a.x + kb * g.sy, at, a.w,
                                                        std::make_integer_sequence<int, rw.n2>{});
        if (!VARNU) c = scaled(a.sc, c);
      }
      v += VARNU ? T(g.eisc[k]) * c : c;
    }
    if constexpr (ROW) a.p[idx] = v;
    else if constexpr (rw.n2 > 0) a.p[idx] = __ldg(x + 3 * G * g.arr) - ml * (bv - v);
    else a.p[idx] -= ml * (bv - v);
  }
}
template <int DISC, int VARNU, class T>
__global__ void __launch_bounds__(kPressThreads, DISC == 2 || sizeof(T) == 8 ? 2 : 3) k_pressure(const __grid_constant__ PressA<T, bc_nw<DISC, VARNU>()> a) {
  press_body<DISC, VARNU, false>(blockIdx, a);
}
template <int DISC, int VARNU, class T>
__global__ void __launch_bounds__(kPressThreads, DISC == 2 || sizeof(T) == 8 ? 2 : 3) kb_pressure(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<PressA<T, bc_nw<DISC, VARNU>()>>(items, n, bid, gd);
  press_body<DISC, VARNU, false>(bid, it.a);
}

template <int DISC, int VARNU>
__global__ void __launch_bounds__(kPressThreads, 2) k_bc(const __grid_constant__ PressA<double, bc_nw<DISC, VARNU>()> a) {
  press_body<DISC, VARNU, true>(blockIdx, a);
}

// P1-P1: the new pressures back into the iterate
template <class T>
struct CopyA { const T* a; T* b; int64_t n; };
template <class T>
__device__ __forceinline__ void copy_body(const uint3 bid, const uint3 gd, const CopyA<T>& c) {
  for (int64_t q = bid.x * int64_t(blockDim.x) + threadIdx.x; q < c.n; q += int64_t(gd.x) * blockDim.x) c.b[q] = c.a[q];
}
template <class T>
__global__ void __launch_bounds__(256) k_copy(const __grid_constant__ CopyA<T> c) {
  copy_body<T>(blockIdx, gridDim, c);
}
template <class T>
__global__ void __launch_bounds__(256) kb_copy(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<CopyA<T>>(items, n, bid, gd);
  copy_body<T>(bid, gd, it.a);
}

template <class A>
void launch(const void* kernel, const void* batched, dim3 grd, int threads, const A& a, cudaStream_t s) {
  if (g_rec) return g_rec->add(batched, grd, dim3(threads), 0, 1, a);
  ++g_launches;
  void* args[] = {const_cast<A*>(&a)};
  cudaLaunchKernel(kernel, grd, dim3(threads), args, 0, s);
}

template <int DISC, int VARNU, class T>
void launch_bt(const Geo& g, int mode, const T* w, const T* x, const T* b, T* y, cudaStream_t s) {
  constexpr int NW = bt_nw<DISC, VARNU>();
  if constexpr (DISC == 1 && sizeof(T) == 4) {
    if (quad_bt(VARNU, g, w, x, mode == MODE_RES ? b : nullptr, y, s)) return;
  }
  BtA<T, NW> a{g, x, mode == MODE_RES ? b : nullptr, y, make_factor<T>(g.h * g.h / row_scale<T>(kScaleB<DISC>)), {}};
  if (NW > 1) std::copy(w, w + NW, a.w);
  const dim3 grd((g.ny * g.sx + kBtThreads - 1) / kBtThreads, g.nz, DISC == 2 ? 3 : 1);
  launch(reinterpret_cast<const void*>(k_bt<DISC, VARNU, T>), reinterpret_cast<const void*>(kb_bt<DISC, VARNU, T>), grd,
         kBtThreads, a, s);
}
// planes of a block: several where the level fills the GPU anyway
int press_planes(const Geo& g) { return int64_t(g.nx + 1) * (g.ny + 1) * (g.nz + 1) > 1000000 ? 4 : 1; }
template <int DISC, int VARNU, class T>
void launch_pressure(const Geo& g, const T* w, const ResTabs<T>* tabs, T* x, const T* b, T* tmp,
                     const double* inv_mlhat, double sc, cudaStream_t s) {
  constexpr int NW = bc_nw<DISC, VARNU>(), G = DISC == 2 ? 8 : 1;
  T* p = x + 3 * G * g.arr;
  const int kp = press_planes(g);
  PressA<T, NW> a{g, x, b, DISC == 2 ? p : tmp + 3 * G * g.arr, inv_mlhat, sc, tabs, kp,
                   make_factor<T>(g.h * g.h / row_scale<T>(kScaleB<DISC>)),
                   make_factor<T>(g.h * g.h * g.h / row_scale<T>(inv_unit_c<VARNU>())), {}};
  if (NW > 1) std::copy(w, w + NW, a.w);
  const dim3 grd((g.ny * g.sx + g.nx + kPressThreads) / kPressThreads, (g.nz + kp) / kp);
  bool done = false;
  if constexpr (DISC == 1 && sizeof(T) == 4) done = quad_pressure(VARNU, g, w, tabs, x, b, a.p, inv_mlhat, sc, s);
  if (!done)
    launch(reinterpret_cast<const void*>(k_pressure<DISC, VARNU, T>),
           reinterpret_cast<const void*>(kb_pressure<DISC, VARNU, T>), grd, kPressThreads, a, s);
  if (DISC == 1)
    launch(reinterpret_cast<const void*>(k_copy<T>), reinterpret_cast<const void*>(kb_copy<T>),
           dim3(unsigned(std::min<int64_t>((g.arr + 255) / 256, 152 * 8))), 256, CopyA<T>{a.p, p, g.arr}, s);
}

template <int DISC, int VARNU>
void launch_bc(const Geo& g, const double* w, const ResTabs<double>* tabs, const double* x, double* y, cudaStream_t s) {
  constexpr int NW = bc_nw<DISC, VARNU>(), G = DISC == 2 ? 8 : 1;
  PressA<double, NW> a{g, x, nullptr, y + 3 * G * g.arr, nullptr, 0.0, tabs, press_planes(g),
                       make_factor<double>(g.h * g.h / row_scale<double>(kScaleB<DISC>)),
                       make_factor<double>(g.h * g.h * g.h / row_scale<double>(inv_unit_c<VARNU>())), {}};
  if (NW > 1) std::copy(w, w + NW, a.w);
  const dim3 grd((g.ny * g.sx + g.nx + kPressThreads) / kPressThreads, (g.nz + a.kp) / a.kp);
  ++g_launches;
  k_bc<DISC, VARNU><<<grd, kPressThreads, 0, s>>>(a);
}

}  // namespace

RowsShape bt_shape(int disc, bool fp32, const Geo& g) {
  if (disc == 1 && fp32 && quad_level(g)) return {kQuadThreads, kQuadPlanes, 4};
  return {kBtThreads, 1, 1};
}
RowsShape pressure_shape(int disc, bool fp32, const Geo& g) {
  if (disc == 1 && fp32 && quad_level(g)) return {kQuadThreads, kQuadPlanes, 4};
  return {kPressThreads, press_planes(g), 1};
}

void bc_rows(int disc, int varnu, const Geo& g, const double* w, const ResTabs<double>* tabs, const double* x,
             double* y, cudaStream_t s) {
  if (disc == 1 && !varnu) launch_bc<1, 0>(g, w, tabs, x, y, s);
  else if (disc == 1) launch_bc<1, 1>(g, w, tabs, x, y, s);
  else if (!varnu) launch_bc<2, 0>(g, w, tabs, x, y, s);
  else launch_bc<2, 1>(g, w, tabs, x, y, s);
}

template <class T>
void bt_rows(int disc, int varnu, int mode, const Geo& g, const T* w, const T* x, const T* b, T* y, cudaStream_t s) {
  if (disc == 1 && !varnu) launch_bt<1, 0, T>(g, mode, w, x, b, y, s);
  else if (disc == 1) launch_bt<1, 1, T>(g, mode, w, x, b, y, s);
  else if (!varnu) launch_bt<2, 0, T>(g, mode, w, x, b, y, s);
  else launch_bt<2, 1, T>(g, mode, w, x, b, y, s);
}

template <class T>
void uzawa_pressure(int disc, int varnu, const Geo& g, const T* w, const ResTabs<T>* tabs, T* x, const T* b, T* tmp,
                    const double* inv_mlhat, double sc, cudaStream_t s) {
  if (disc == 1 && !varnu) launch_pressure<1, 0, T>(g, w, tabs, x, b, tmp, inv_mlhat, sc, s);
  else if (disc == 1) launch_pressure<1, 1, T>(g, w, tabs, x, b, tmp, inv_mlhat, sc, s);
  else if (!varnu) launch_pressure<2, 0, T>(g, w, tabs, x, b, tmp, inv_mlhat, sc, s);
  else launch_pressure<2, 1, T>(g, w, tabs, x, b, tmp, inv_mlhat, sc, s);
}

#define HHG_INST(T)                                                                                                   \
  template void bt_rows<T>(int, int, int, const Geo&, const T*, const T*, const T*, T*, cudaStream_t);                \
  template void uzawa_pressure<T>(int, int, const Geo&, const T*, const ResTabs<T>*, T*, const T*, T*, const double*, \
                                  double, cudaStream_t);
HHG_INST(double)
HHG_INST(float)

}  // namespace hhg
