// The rows of the P2-P1 operator (apply and residual, FP32) on large levels: a
// thread owns a position of the (i, j) plane and marches along k with its
// stencil footprint in registers.
//
// The rows of one pass (the eight group rows of a velocity component and the
// component's part of the pressure row) read, per site, values of a few
// columns (array, di, dj) at up to three planes each.  A column's planes stay
// in registers while the thread marches, so that a step loads one value per
// column (47 instead of 84) straight from L1/L2 and applies each value to
// every term that reads it (290).  No shared memory, no barriers: a step is
// loads, FMAs with immediate (constant viscosity) or constant-bank weights and
// register moves.  One thread per 32-byte sector prefetches the planes of a
// later step into L2, and the right-hand side is loaded ahead of the sums.
//
// One launch per component (the pressure row's first pass writes it, the later
// ones add to it); the grid is one wave of blocks, runs of planes cut evenly.
//
// Bound: instruction issue (about 690 instructions per site and pass, 290 of
// them FMAs) and the latency of a step's loads at 16 warps per SM.  Measured,
// level 7, 6-tetrahedron cube: apply 206 us (four sites staged in shared
// memory, the kernel this replaces: 271 us), residual 241 us (461 us), with a
// variable viscosity 245 us (314 us).  On level 6 the rows
// without marching (rows.cu) are faster (29 against 41 us): the runs of planes
// are too short to fill the GPU.  P1-P1, with 28 columns
// and 112 or 150 terms, is slower this way than staged (one component's loads
// in flight are too few): it keeps the streaming kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "at.h"
#include "batch.h"
#include "fast.h"
#include "march.h"
#include "structure.inc"

namespace hhg {
namespace {

struct NoTab {};                                   // constant viscosity: no run-time weights
template <int DISC, int VARNU, class T>
using RowTab = std::conditional_t<VARNU != 0, FastTab<T, gen::S<DISC, VARNU, OP_FULL>::N>, NoTab>;

template <class T>
struct MarchA { Geo g; const T* x; const T* b; T* y; int kc; };

// columns of a pass: array slot, i and j offset, the planes lo .. hi read, and
// the first of the column's registers
struct Col { int slot, dj, di, lo, hi, reg; };
template <int MAX>
struct ColTab { int n, nreg; Col c[MAX]; };
template <class SPT, int Q>
constexpr auto make_cols() {
  constexpr gen::PassT ps = SPT::passes[Q];
  ColTab<ps.nl * 3> t{};
  for (int l = ps.l0; l < ps.l0 + ps.nl; ++l)
    for (int e = SPT::lines[l].e0; e < SPT::lines[l].e0 + SPT::lines[l].ne; ++e) {
      const int slot = SPT::lines[l].slot, dj = SPT::lines[l].dj, dk = SPT::lines[l].dk, di = SPT::terms[e].di;
      int q = 0;
      while (q < t.n && !(t.c[q].slot == slot && t.c[q].dj == dj && t.c[q].di == di)) ++q;
      if (q == t.n) {
        t.c[q] = Col{slot, dj, di, dk, dk, 0};
        ++t.n;
      } else {
        if (dk < t.c[q].lo) t.c[q].lo = dk;
        if (dk > t.c[q].hi) t.c[q].hi = dk;
      }
    }
  for (int q = 0; q < t.n; ++q) {
    t.c[q].reg = t.nreg;
    t.nreg += t.c[q].hi - t.c[q].lo + 1;
  }
  return t;
}
template <class SPT, int Q>
struct Cols {
  static constexpr auto t = make_cols<SPT, Q>();
  static constexpr int reg(int slot, int dj, int di, int dk) {
    for (int q = 0; q < t.n; ++q)
      if (t.c[q].slot == slot && t.c[q].dj == dj && t.c[q].di == di) return t.c[q].reg + dk - t.c[q].lo;
    return -1;
  }
};

template <class SPT, int E, int VARNU, class T, class Tab>
__device__ __forceinline__ T mweight(const Tab& tab) {
  if constexpr (VARNU) {
    return tab.w[E];
  } else {
    constexpr double w = SPT::wref[E];
    return T(w);
  }
}

// column C's value at plane offset dk from site i (P2-P1 and constant
// viscosity: pressure values scaled by h as loaded)
template <class SPT, int Q, int C, int PARR, int VARNU, int DK, class T>
__device__ __forceinline__ T col_load(const Geo& g, const T* __restrict__ x, const Lines<T>& at, T hs) {
  constexpr Col c = Cols<SPT, Q>::t.c[C];
  constexpr int arr = SPT::arrs[SPT::passes[Q].a0 + c.slot];
  const T v = at.template ld<c.di, c.dj, DK>(x + arr * g.arr);
  return !VARNU && arr == PARR ? hs * v : v;
}
template <class SPT, int Q, int PARR, int VARNU, class T, int NR, int... C>
__device__ __forceinline__ void first_loads(const Geo& g, const T* x, const Lines<T>& at, T hs, T (&w)[NR],
                                            std::integer_sequence<int, C...>) {
  ([&] {
    constexpr Col c = Cols<SPT, Q>::t.c[C];
    if constexpr (c.lo < c.hi) w[c.reg] = col_load<SPT, Q, C, PARR, VARNU, c.lo>(g, x, at, hs);
    if constexpr (c.lo + 1 < c.hi) w[c.reg + 1] = col_load<SPT, Q, C, PARR, VARNU, c.lo + 1>(g, x, at, hs);
  }(), ...);
}
template <class SPT, int Q, int PARR, int VARNU, class T, int NR, int... C>
__device__ __forceinline__ void step_loads(const Geo& g, const T* x, const Lines<T>& at, T hs, T (&w)[NR],
                                           std::integer_sequence<int, C...>) {
  ([&] {
    constexpr Col c = Cols<SPT, Q>::t.c[C];
    w[c.reg + c.hi - c.lo] = col_load<SPT, Q, C, PARR, VARNU, c.hi>(g, x, at, hs);
  }(), ...);
}
template <class SPT, int Q, class T, int NR, int... C>
__device__ __forceinline__ void shift(T (&w)[NR], std::integer_sequence<int, C...>) {
  ([&] {
    constexpr Col c = Cols<SPT, Q>::t.c[C];
#pragma unroll
    for (int d = 0; d < c.hi - c.lo; ++d) w[c.reg + d] = w[c.reg + d + 1];
  }(), ...);
}

// acc[2 part + segment] (constant viscosity: the segments B^T and A share one)
template <class SPT, int Q, int L, int VARNU, class T, class Tab, int NR, int NA, int... I>
__device__ __forceinline__ void line_terms(const T (&w)[NR], T (&acc)[NA], const Tab& tab,
                                           std::integer_sequence<int, I...>) {
  ([&] {
    constexpr gen::LineT ln = SPT::lines[L];
    constexpr gen::TermE te = SPT::terms[ln.e0 + I];
    constexpr int a = 2 * te.part + (VARNU ? te.seg : 0), r = Cols<SPT, Q>::reg(ln.slot, ln.dj, te.di, ln.dk);
    acc[a] = fma(mweight<SPT, te.t, VARNU, T>(tab), w[r], acc[a]);
  }(), ...);
}
template <class SPT, int Q, int VARNU, class T, class Tab, int NR, int NA, int... L>
__device__ __forceinline__ void all_terms(const T (&w)[NR], T (&acc)[NA], const Tab& tab,
                                          std::integer_sequence<int, L...>) {
  (line_terms<SPT, Q, SPT::passes[Q].l0 + L, VARNU>(
       w, acc, tab, std::make_integer_sequence<int, SPT::lines[SPT::passes[Q].l0 + L].ne>{}), ...);
}

// what the rows of a step are combined with -- the right-hand side (MODE_RES),
// or the row so far (later passes of the pressure row) -- loaded ahead of the
// step's sums
template <int DISC, int VARNU, int MODE, int Q, class T, int NP, int... P>
__device__ __forceinline__ void old_values(const MarchA<T>& a, unsigned at, T (&old)[NP],
                                           std::integer_sequence<int, P...>) {
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  ([&] {
    constexpr gen::PartT pt = SPT::parts[SPT::passes[Q].p0 + P];
    if constexpr (!pt.first) old[P] = ref_at(a.y + pt.out * a.g.arr, at);
    else if constexpr (MODE == MODE_RES) old[P] = ld_at(a.b + pt.out * a.g.arr, at);
  }(), ...);
}
// the pass's input planes (and right-hand side) at site `at` into L2
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
template <int DISC, int VARNU, int MODE, int Q, class T, int... A>
__device__ __forceinline__ void prefetch_planes(const MarchA<T>& a, unsigned at, std::integer_sequence<int, A...>) {
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  ([&] {
    constexpr int arr = SPT::arrs[SPT::passes[Q].a0 + A];
    prefetch_l2(reinterpret_cast<const char*>(a.x + arr * a.g.arr) + at);
    if (MODE == MODE_RES) prefetch_l2(reinterpret_cast<const char*>(a.b + arr * a.g.arr) + at);
  }(), ...);
}

template <int DISC, int VARNU, int MODE, int Q, class T, int NA, int NP, int... P>
__device__ __forceinline__ void store_rows(const MarchA<T>& a, int i, int j, int k, unsigned at, const T (&acc)[NA],
                                           const T (&old)[NP], std::integer_sequence<int, P...>) {
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  static_assert(gen::S<DISC, VARNU, OP_FULL>::rows[24].n2 == 0, "P2-P1: no C terms");
  const Geo& g = a.g;
  const T es = VARNU ? T(__ldg(g.esc + k)) : T(1);
  ([&] {
    constexpr gen::PartT pt = SPT::parts[SPT::passes[Q].p0 + P];
    constexpr int ox = (0xB2 >> pt.og) & 1, oy = (0xD4 >> pt.og) & 1, oz = (0xE8 >> pt.og) & 1;
    if (i <= g.nx - ox && j <= g.ny - oy && k <= g.nz - oz) {
      const bool inside = (ox || (i > 0 && i < g.nx)) && (oy || (j > 0 && j < g.ny)) && (oz || (k > 0 && k < g.nz));
      const T v = VARNU ? acc[2 * P] + es * acc[2 * P + 1] : (pt.all ? T(g.h) * T(g.h) : T(g.h)) * acc[2 * P];
      T& y = ref_at(a.y + pt.out * g.arr, at);
      if (!pt.all && !inside) {
        y = T(0);                              // Dirichlet velocity row
      } else if (pt.first) {
        y = MODE == MODE_RES ? old[P] - v : v;
      } else {
        y = MODE == MODE_RES ? old[P] - v : old[P] + v;
      }
    }
  }(), ...);
}

constexpr int kAhead = 4;                          // planes between a prefetch and its use

// grid x over the positions of the padded (i, j) plane, y = runs of kc planes
template <int DISC, int VARNU, int MODE, int Q, class T, class Tab>
__device__ __forceinline__ void march_body(const uint3 bid, const MarchA<T>& a, const Tab& tab) {
  using SPT = gen::SP<DISC, VARNU, OP_FULL>;
  constexpr gen::PassT ps = SPT::passes[Q];
  constexpr auto cols = std::make_integer_sequence<int, Cols<SPT, Q>::t.n>{};
  constexpr int PARR = 24;
  const Geo& g = a.g;
  const int q = bid.x * blockDim.x + threadIdx.x, j = q / g.sx, i = q - j * g.sx;
  if (i > g.nx || j > g.ny) return;
  const int k0 = bid.y * a.kc, k1 = min(k0 + a.kc, g.nz + 1);
  const unsigned plane = unsigned(g.sy);
  unsigned site = unsigned(i + 1 + (j + 1) * g.sx) + unsigned(k0 + 1) * plane;
  const T hs = T(g.h);
  T w[Cols<SPT, Q>::t.nreg];
  first_loads<SPT, Q, PARR, VARNU>(g, a.x, Lines<T>(g, site), hs, w, cols);
#pragma unroll 1
  for (int k = k0; k < k1; ++k, site += plane) {
    const Lines<T> lines(g, site);
    const unsigned at = lines.site();
    step_loads<SPT, Q, PARR, VARNU>(g, a.x, lines, hs, w, cols);
    T old[ps.np], acc[2 * ps.np] = {};
    old_values<DISC, VARNU, MODE, Q>(a, at, old, std::make_integer_sequence<int, ps.np>{});
    if ((threadIdx.x & 7) == 0 && k + kAhead < k1)  // one thread per 32-byte sector
      prefetch_planes<DISC, VARNU, MODE, Q>(a, at + kAhead * plane * unsigned(sizeof(T)), std::make_integer_sequence<int, ps.na>{});
    all_terms<SPT, Q, VARNU>(w, acc, tab, std::make_integer_sequence<int, ps.nl>{});
    store_rows<DISC, VARNU, MODE, Q>(a, i, j, k, at, acc, old, std::make_integer_sequence<int, ps.np>{});
    shift<SPT, Q>(w, cols);
  }
}
constexpr int kMarchThreads = 256;
template <int DISC, int VARNU, int MODE, int Q, class T>
__global__ void __launch_bounds__(kMarchThreads, 2)
    k_march(const __grid_constant__ MarchA<T> a, const __grid_constant__ RowTab<DISC, VARNU, T> tab) {
  march_body<DISC, VARNU, MODE, Q>(blockIdx, a, tab);
}
template <int DISC, int VARNU, class T>
struct MarchB { MarchA<T> a; const RowTab<DISC, VARNU, T>* tab; };
template <int DISC, int VARNU, int MODE, int Q, class T>
__global__ void __launch_bounds__(kMarchThreads, 2) kb_march(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<MarchB<DISC, VARNU, T>>(items, n, bid, gd);
  march_body<DISC, VARNU, MODE, Q>(bid, it.a.a, *it.a.tab);
}

template <int DISC, int VARNU, int MODE, class T, int... Q>
void launch_march(MarchA<T>& a, const void* tab, cudaStream_t s, std::integer_sequence<int, Q...>) {
  using Tab = RowTab<DISC, VARNU, T>;
  const Geo& g = a.g;
  const int nb = (g.ny * g.sx + g.nx + kMarchThreads) / kMarchThreads;
  const int runs = std::max(1, std::min(2 * 152 / nb, (g.nz + 8) / 8));
  a.kc = (g.nz + runs) / runs;
  const dim3 grd(nb, (g.nz + a.kc) / a.kc);
  const Tab none{};
  const void* t = VARNU ? tab : static_cast<const void*>(&none);
  ([&] {
    if (g_rec) {
      const Tab* dt = VARNU ? static_cast<const Tab*>(g_rec->table(tab, sizeof(Tab))) : nullptr;
      g_rec->add(reinterpret_cast<const void*>(kb_march<DISC, VARNU, MODE, Q, T>), grd, dim3(kMarchThreads), 0, 1,
                 MarchB<DISC, VARNU, T>{a, dt});
    } else {
      ++g_launches;
      void* args[] = {&a, const_cast<void*>(t)};
      cudaLaunchKernel(reinterpret_cast<const void*>(k_march<DISC, VARNU, MODE, Q, T>), grd, dim3(kMarchThreads), args,
                       0, s);
    }
  }(), ...);
}

}  // namespace

template <class T>
void march_rows(int varnu, int mode, const Geo& g, const void* tab, const T* x, const T* b, T* y, cudaStream_t s) {
  MarchA<T> a{g, x, b, y, 1};
  auto launch = [&](auto v) {
    constexpr int V = decltype(v)::value;
    using Passes = std::make_integer_sequence<int, gen::SP<2, V, OP_FULL>::NP>;
    if (mode == MODE_RES) launch_march<2, V, MODE_RES, T>(a, tab, s, Passes{});
    else launch_march<2, V, MODE_SET, T>(a, tab, s, Passes{});
  };
  if (varnu) launch(std::integral_constant<int, 1>{});
  else launch(std::integral_constant<int, 0>{});
}
template void march_rows<float>(int, int, const Geo&, const void*, const float*, const float*, float*, cudaStream_t);

}  // namespace hhg
