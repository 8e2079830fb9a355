// The rows of the full operator (apply and residual) on levels too small for
// the streaming kernels (stream.cu).
//
// P2-P1: a thread owns a lattice site and a velocity component and evaluates
// all eight group rows there, input value by input value: each of the ~120
// values the eight rows read is loaded once and applied to every row that
// reads it (238 terms), in registers; other threads take the pressure row
// (156 terms).  P1-P1: a thread evaluates the three velocity rows of a site,
// another one the pressure row.  The terms
// are unrolled from the generated plan; with a constant viscosity the weights
// are immediates (those of h = 1, the segments of a row scaled at the end),
// with a variable one they come from the constant bank.  Boundary pressure rows keep the merged B terms (exact for
// zero Dirichlet velocities) and take the C stencil of their boundary class.
//
// Bound: launch latency on the smallest levels, the L1 loads at level 6.
// Measured against the kernels this replaces (a thread per row and site, or
// four sites, with a weight and an offset of every term from the constant
// bank, and a serial loop over cubes for the C terms of boundary rows), the
// residual in FP32 P2-P1, level 3 / 5 / 6: 20.6 / 21.5 / 71.8 us before, 6.3 /
// 8.3 / 39.0 us now; FP64 P1-P1, level 4: 14.4 us before, 6.2 us.
#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

#include "at.h"
#include "batch.h"
#include "fast.h"
#include "rows.h"
#include "structure.inc"
#include "weights.h"

namespace hhg {
namespace {

// whether the rows take the level's weights from a table; FP64 P1-P1 does so
// with a constant viscosity too (few weights, and the coarse matrix, whose
// rows these are, keeps the level's stencils to the last bit)
template <int DISC, int VARNU, class T>
constexpr bool kTabled = VARNU != 0 || (DISC == 1 && sizeof(T) == 8);
struct NoTab {};
template <int DISC, int VARNU, class T>
using RowTab = std::conditional_t<kTabled<DISC, VARNU, T>, FastTab<T, gen::S<DISC, VARNU, OP_FULL>::N>, NoTab>;

// h and h^2 in T.  FP32: where they are not exact, in two parts (weights.h; a
// rounded factor would be a relative error of up to 6e-8 common to all rows).
template <class T>
struct Powers { Factor<T> h, h2; bool inexact; };
template <class T>
Powers<T> make_powers(double h) {
  if (sizeof(T) == 8 || (T(h) == h && T(h * h) == h * h)) return {{T(h), T(0)}, {T(h * h), T(0)}, false};
  return {make_factor<T>(h), make_factor<T>(h * h), true};
}
// h^2 times a sum of B^T plus h times one of A
template <class T>
__device__ __forceinline__ T combine(const Powers<T>& h, T bt, T a) {
  if constexpr (sizeof(T) == 8) return fma(h.h.hi, a, h.h2.hi * bt);
  const T low = h.inexact ? fma(h.h2.lo, bt, h.h.lo * a) : T(0);
  return fma(h.h.hi, a, fma(h.h2.hi, bt, low));
}

template <class T>
struct FullA { Geo g; const T* x; const T* b; T* y; const ResTabs<T>* tabs; Powers<T> h; };

template <class SPT, int T0, class T, class Tab>
__device__ __forceinline__ T fweight(const Tab& tab) {
  if constexpr (!std::is_same<Tab, NoTab>::value) {
    return tab.w[T0];
  } else {
    constexpr double w = SPT::wref[T0];
    return T(w);
  }
}

// whether line L has a term at i offset DI, in a velocity row (VEL) or any row
template <class SPT, int L, int DI, bool VEL>
constexpr bool line_reads(int p0) {
  for (int e = SPT::lines[L].e0; e < SPT::lines[L].e0 + SPT::lines[L].ne; ++e)
    if (SPT::terms[e].di == DI && !(VEL && SPT::parts[p0 + SPT::terms[e].part].all)) return true;
  return false;
}

// the terms of line L at i offset DI applied to the accumulators acc[2 part +
// segment] of the pass's rows (B^T and A apart)
template <class SPT, int Q, int L, int DI, bool VEL, class T, class Tab, int NA, int... I>
__device__ __forceinline__ void line_value(T v, T (&acc)[NA], const Tab& tab, std::integer_sequence<int, I...>) {
  ([&] {
    constexpr int e = SPT::lines[L].e0 + I;
    constexpr gen::TermE te = SPT::terms[e];
    if constexpr (te.di == DI && te.seg < 2 && !(VEL && SPT::parts[SPT::passes[Q].p0 + te.part].all)) {
      constexpr int a = 2 * te.part + te.seg;
      acc[a] = fma(fweight<SPT, te.t, T>(tab), v, acc[a]);
    }
  }(), ...);
}
template <class SPT, int Q, int L, bool VEL, class T, class Tab, int NA>
__device__ __forceinline__ void one_line(const Geo& g, const T* __restrict__ x, const Lines<T>& at, T (&acc)[NA],
                                         const Tab& tab) {
  constexpr gen::LineT ln = SPT::lines[L];
  constexpr int arr = SPT::arrs[SPT::passes[Q].a0 + ln.slot];
  const T* p = x + arr * g.arr;
  const auto all = std::make_integer_sequence<int, ln.ne>{};
  constexpr int p0 = SPT::passes[Q].p0;
  if constexpr (line_reads<SPT, L, -1, VEL>(p0)) line_value<SPT, Q, L, -1, VEL>(at.template ld<-1, ln.dj, ln.dk>(p), acc, tab, all);
  if constexpr (line_reads<SPT, L, 0, VEL>(p0)) line_value<SPT, Q, L, 0, VEL>(at.template ld<0, ln.dj, ln.dk>(p), acc, tab, all);
  if constexpr (line_reads<SPT, L, 1, VEL>(p0)) line_value<SPT, Q, L, 1, VEL>(at.template ld<1, ln.dj, ln.dk>(p), acc, tab, all);
}
template <class SPT, int Q, bool VEL, class T, class Tab, int NA, int... L>
__device__ __forceinline__ void all_lines(const Geo& g, const T* __restrict__ x, const Lines<T>& at, T (&acc)[NA],
                                          const Tab& tab,
                                          std::integer_sequence<int, L...>) {
  (one_line<SPT, Q, SPT::passes[Q].l0 + L, VEL>(g, x, at, acc, tab), ...);
}

// interior C terms of the pressure row (segment 2), weights w of the level
// (|T|^(2/3) does not scale exactly from h = 1)
template <class S, int T0, class T, int... I>
__device__ __forceinline__ T c_terms(const Geo& g, const T* __restrict__ x, const Lines<T>& at, const T* __restrict__ w,
                                     std::integer_sequence<int, I...>) {
  T a = T(0);
  ([&] {
    constexpr gen::OffT o = S::off[T0 + I];
    a = fma(__ldg(w + I), at.template ld<o.di, o.dj, o.dk>(x + o.arr * g.arr), a);
  }(), ...);
  return a;
}
// place in the table of the I-th of n terms of an FP32 row of A: the diagonal,
// first in the table, comes in the middle, where it meets half of the terms that
// cancel it (error of a 7-term row on smooth fields 2.3e-7, in table order up to
// 4.1e-7)
constexpr int diag_middle(int I, int n) { return I < n / 2 ? I + 1 : I == n / 2 ? 0 : I; }
// terms [T0, T0 + n) of a row: one chain
template <class S, int T0, int SEG, class SPT, class T, class Tab, int... I>
__device__ __forceinline__ T chain(const Geo& g, const T* __restrict__ x, const Lines<T>& at, const Tab& tab,
                                   std::integer_sequence<int, I...>) {
  T a = T(0);
  ([&] {
    constexpr int e = T0 + (SEG == 1 && sizeof(T) == 4 ? diag_middle(I, sizeof...(I)) : I);
    constexpr gen::OffT o = S::off[e];
    a = fma(fweight<SPT, e, T>(tab), at.template ld<o.di, o.dj, o.dk>(x + o.arr * g.arr), a);
  }(), ...);
  return a;
}
// terms [T0, T0 + n) of the pressure row: eight (P1-P1: three, a component each)
// chains of consecutive terms (FP32 error of the apply's pressure, P2-P1 level 6:
// 1.9e-7 in one chain, 4.8e-7 with the terms dealt out to four in turn, 1.0e-7
// now; see chain_of)
template <int DISC, class S, int T0, class SPT, class T, class Tab, int... I>
__device__ __forceinline__ T b_terms(const Geo& g, const T* __restrict__ x, const Lines<T>& at, const Tab& tab,
                                     std::integer_sequence<int, I...>) {
  constexpr int M = DISC == 2 ? 8 : 3;
  T a[M] = {};
  ([&] {
    constexpr gen::OffT o = S::off[T0 + I];
    constexpr int q = chain_of(I, sizeof...(I), M);
    a[q] = fma(fweight<SPT, T0 + I, T>(tab), at.template ld<o.di, o.dj, o.dk>(x + o.arr * g.arr), a[q]);
  }(), ...);
  if constexpr (M == 3) return (a[0] + a[1]) + a[2];
  else return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

template <int MODE, class T>
__device__ __forceinline__ void put(const FullA<T>& a, int arr, unsigned i, bool inside, T v) {
  T& y = ref_at(a.y + int64_t(arr) * a.g.arr, i);
  if (MODE == MODE_RES) y = inside ? ld_at(a.b + int64_t(arr) * a.g.arr, i) - v : T(0);
  else y = inside ? v : T(0);
}

// the velocity rows of pass Q (a component; P1: all three) at site (i, j, k)
template <int DISC, int VARNU, int MODE, int Q, class T, class Tab, int... P>
__device__ __forceinline__ void velocity_rows(const FullA<T>& a, int i, int j, int k, const Lines<T>& at, const Tab& tab,
                                              std::integer_sequence<int, P...>) {
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  constexpr gen::PassT ps = SPT::passes[Q];
  const Geo& g = a.g;
  T acc[2 * ps.np] = {};
  all_lines<SPT, Q, true>(g, a.x, at, acc, tab, std::make_integer_sequence<int, ps.nl>{});
  // the segments' scales: B^T unscaled (weights at h = 1: h^2), A exp(nu_a h k) (h)
  constexpr bool tabled = kTabled<DISC, VARNU, T>;
  const T es = VARNU ? T(g.esc[k]) : T(1);
  ([&] {
    constexpr gen::PartT pt = SPT::parts[ps.p0 + P];
    if constexpr (!pt.all) {
      constexpr int ox = (0xB2 >> pt.og) & 1, oy = (0xD4 >> pt.og) & 1, oz = (0xE8 >> pt.og) & 1;
      if (i <= g.nx - ox && j <= g.ny - oy && k <= g.nz - oz) {
        const bool inside = (ox || (i > 0 && i < g.nx)) && (oy || (j > 0 && j < g.ny)) && (oz || (k > 0 && k < g.nz));
        put<MODE>(a, pt.out, at.site(), inside,
                  tabled ? acc[2 * P] + es * acc[2 * P + 1] : combine(a.h, acc[2 * P], acc[2 * P + 1]));
      }
    }
  }(), ...);
}

// P1-P1: the velocity rows, row by row (a row's B^T and A segments one chain each; the components' pressure loads are the same)
template <int VARNU, int MODE, class T, class Tab, int... R>
__device__ __forceinline__ void velocity_rows_p1(const FullA<T>& a, int i, int j, int k, const Lines<T>& at,
                                                 const Tab& tab, std::integer_sequence<int, R...>) {
  using S = gen::S<1, VARNU, OP_FULL>;
  using SPT = gen::SP<1, VARNU, OP_FULL>;
  const Geo& g = a.g;
  constexpr bool tabled = kTabled<1, VARNU, T>;
  const T es = VARNU ? T(g.esc[k]) : T(1);
  const bool inside = i > 0 && i < g.nx && j > 0 && j < g.ny && k > 0 && k < g.nz;
  ([&] {
    constexpr gen::RowS rw = S::rows[R];
    static_assert(rw.n2 == 0, "no C terms in a velocity row");
    const T a0 = chain<S, rw.t0, 0, SPT>(g, a.x, at, tab, std::make_integer_sequence<int, rw.n0>{});
    const T a1 = chain<S, rw.t0 + rw.n0, 1, SPT>(g, a.x, at, tab, std::make_integer_sequence<int, rw.n1>{});
    put<MODE>(a, rw.out, at.site(), inside, tabled ? a0 + es * a1 : combine(a.h, a0, a1));
  }(), ...);
}

template <int DISC, int VARNU, int MODE, class T, class Tab>
__device__ __forceinline__ void pressure_row(const FullA<T>& a, int i, int j, int k, const Lines<T>& at, const Tab& tab) {
  using S = gen::S<DISC, VARNU, OP_FULL>;
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  constexpr int PARR = DISC == 2 ? 24 : 3;
  constexpr gen::RowS rw = S::rows[PARR];
  static_assert(rw.out == PARR && rw.n1 == 0, "the last row is the pressure's; B is unscaled");
  const Geo& g = a.g;
  T v = b_terms<DISC, S, rw.t0, SPT>(g, a.x, at, tab, std::make_integer_sequence<int, rw.n0>{});
  if (!kTabled<DISC, VARNU, T>) v = a.h.inexact ? scaled(a.h.h2, v) : a.h.h2.hi * v;
  if constexpr (rw.n2 > 0) {
    T c;
    if (i == 0 || j == 0 || k == 0 || i == g.nx || j == g.ny || k == g.nz) {
      const int cls = (i == 0 ? 0 : i == g.nx ? 2 : 1) + 3 * (j == 0 ? 0 : j == g.ny ? 2 : 1) +
                      9 * (k == 0 ? 0 : k == g.nz ? 2 : 1);
      c = c_class<SPT>(g, a.x + PARR * g.arr + at.site() / unsigned(sizeof(T)), a.tabs->wc + cls * SPT::NCB, std::make_integer_sequence<int, SPT::NCB>{});
    } else {
      using SBC = gen::S<DISC, VARNU, OP_BC>;
      constexpr int wc0 = gen::S<DISC, VARNU, OP_A>::N / 3 + gen::S<DISC, VARNU, OP_BT>::N + SBC::rows[0].n0;
      static_assert(SBC::rows[0].n1 == 0 && SBC::rows[0].n2 == rw.n2, "the row of (B, -C) is the full operator's");
      c = c_terms<S, rw.t0 + rw.n0>(g, a.x, at, a.tabs->w + wc0, std::make_integer_sequence<int, rw.n2>{});
    }
    v += VARNU ? T(g.eisc[k]) * c : c;
  }
  put<MODE>(a, PARR, at.site(), true, v);
}

// grid x over the sites of the (i, j) plane (flat), y = plane, z = part: P1-P1 the
// components, all at once, then the pressure; P2-P1 the pressure, whose row is
// the longest chain of sums, then the components
template <int DISC, int VARNU, int MODE, class T, class Tab>
__device__ __forceinline__ void full_body(const uint3 bid, const FullA<T>& full, const Tab& tab) {
  const Geo& g = full.g;
  const int w = g.nx + 1, q = bid.x * blockDim.x + threadIdx.x, j = q / w, i = q - j * w, k = bid.y;
  if (j > g.ny) return;
  const int kb = kByPlane<DISC, T> ? k : 0;          // the plane that offsets count from
  const FullA<T> a{g, full.x + kb * g.sy, full.b + kb * g.sy, full.y + kb * g.sy, full.tabs, full.h};
  const Lines<T> at(g, unsigned(i + 1) + unsigned(j + 1) * unsigned(g.sx) + unsigned(k - kb + 1) * unsigned(g.sy));
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  if constexpr (DISC == 1) {
    if (bid.z == 0)
      velocity_rows_p1<VARNU, MODE>(a, i, j, k, at, tab, std::make_integer_sequence<int, 3>{});
    else
      pressure_row<1, VARNU, MODE>(a, i, j, k, at, tab);
  } else {
    if (bid.z == 1)
      velocity_rows<2, VARNU, MODE, 0>(a, i, j, k, at, tab, std::make_integer_sequence<int, SPT::passes[0].np>{});
    else if (bid.z == 2)
      velocity_rows<2, VARNU, MODE, 1>(a, i, j, k, at, tab, std::make_integer_sequence<int, SPT::passes[1].np>{});
    else if (bid.z == 3)
      velocity_rows<2, VARNU, MODE, 2>(a, i, j, k, at, tab, std::make_integer_sequence<int, SPT::passes[2].np>{});
    else
      pressure_row<2, VARNU, MODE>(a, i, j, k, at, tab);
  }
}
template <int DISC, int VARNU, int MODE, class T>
__global__ void __launch_bounds__(128) k_full(const __grid_constant__ FullA<T> a,
                                              const __grid_constant__ RowTab<DISC, VARNU, T> tab) {
  full_body<DISC, VARNU, MODE>(blockIdx, a, tab);
}
// batched: the table as a device copy, read through the uniform path
template <int DISC, int VARNU, class T>
struct FullB { FullA<T> a; const RowTab<DISC, VARNU, T>* tab; };
template <int DISC, int VARNU, int MODE, class T>
__global__ void __launch_bounds__(128) kb_full(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<FullB<DISC, VARNU, T>>(items, n, bid, gd);
  full_body<DISC, VARNU, MODE>(bid, it.a.a, *it.a.tab);
}

template <int DISC, int VARNU, int MODE, class T>
void launch_full(const FullA<T>& a, const void* tab, cudaStream_t s) {
  using Tab = RowTab<DISC, VARNU, T>;
  const Geo& g = a.g;
  const dim3 grd(((g.nx + 1) * (g.ny + 1) + 127) / 128, g.nz + 1, DISC == 2 ? 4 : 2);
  constexpr bool tabled = kTabled<DISC, VARNU, T>;
  const NoTab none{};
  const void* t = tabled ? tab : static_cast<const void*>(&none);
  if (g_rec) {
    const Tab* dt = tabled ? static_cast<const Tab*>(g_rec->table(tab, sizeof(Tab))) : nullptr;
    return g_rec->add(reinterpret_cast<const void*>(kb_full<DISC, VARNU, MODE, T>), grd, dim3(128), 0, 1,
                      FullB<DISC, VARNU, T>{a, dt});
  }
  ++g_launches;
  void* args[] = {const_cast<FullA<T>*>(&a), const_cast<void*>(t)};
  cudaLaunchKernel(reinterpret_cast<const void*>(k_full<DISC, VARNU, MODE, T>), grd, dim3(128), args, 0, s);
}

}  // namespace

int fast_terms(int disc, int varnu, int op) {
#define HHG_N(D, V, O) if (disc == D && varnu == V && op == O) return gen::S<D, V, O>::N;
  HHG_N(1, 0, OP_FULL) HHG_N(1, 0, OP_A) HHG_N(1, 0, OP_BT) HHG_N(1, 0, OP_BC)
  HHG_N(1, 1, OP_FULL) HHG_N(1, 1, OP_A) HHG_N(1, 1, OP_BT) HHG_N(1, 1, OP_BC)
  HHG_N(2, 0, OP_FULL) HHG_N(2, 0, OP_A) HHG_N(2, 0, OP_BT) HHG_N(2, 0, OP_BC)
  HHG_N(2, 1, OP_FULL) HHG_N(2, 1, OP_A) HHG_N(2, 1, OP_BT) HHG_N(2, 1, OP_BC)
#undef HHG_N
  return -1;
}

template <class T>
void full_rows(int disc, int varnu, int mode, const Geo& g, const void* tab, const ResTabs<T>* tabs, const T* x,
               const T* b, T* y, cudaStream_t s) {
  const FullA<T> a{g, x, b, y, tabs, make_powers<T>(g.h)};
#define HHG_F(D, V)                                                           \
  if (disc == D && varnu == V)                                                \
    return mode == MODE_RES ? launch_full<D, V, MODE_RES, T>(a, tab, s)       \
                            : launch_full<D, V, MODE_SET, T>(a, tab, s);
  HHG_F(1, 0) HHG_F(1, 1) HHG_F(2, 0) HHG_F(2, 1)
#undef HHG_F
}

template void full_rows<double>(int, int, int, const Geo&, const void*, const ResTabs<double>*, const double*,
                                const double*, double*, cudaStream_t);
template void full_rows<float>(int, int, int, const Geo&, const void*, const ResTabs<float>*, const float*,
                               const float*, float*, cudaStream_t);

}  // namespace hhg
