// Shared-memory-resident inexact Uzawa smoother for the small levels of the
// hierarchy (Sec. 3.2, Eqs. uzawa-velocity / uzawa-pressure).
//
// On the coarse levels of a V-cycle every phase of the smoother (the B^T
// residual, each Gauss-Seidel colour or edge group, the (B, -C) residual and
// the pressure update) touches only a few thousand DoFs, so one kernel launch
// per phase costs far more than the arithmetic.  Here one launch of a
// thread-block cluster of C CTAs (1 <= C <= 16) runs all phases of all
// requested Uzawa iterations with the level's block vector in shared memory:
//
//  * CTA c owns the k planes [c (nz+1) / C, (c+1) (nz+1) / C) of every array
//    and stores them, plus one halo plane below and above, site by site: the
//    3G+1 values of a lattice site lie side by side, with an odd stride, so
//    that array and i offset of a stencil term are an immediate of its load
//    (two registers hold the j and k pitch) and the lanes of a warp, which
//    take consecutive sites, hit different banks;
//  * a phase updates the CTA's own sites from shared memory; a value on a
//    boundary plane is also stored into the neighbour's halo plane
//    (distributed shared memory), and a cluster barrier ends the phase;
//  * rows are unrolled from the generated structure: with a constant
//    viscosity the weights are immediates too (the row scaled at the end:
//    weights.h), with a variable one they are read from a shared table;
//  * the right-hand sides tmp_u = b_u - B^T p stay in shared memory.
//
// The vertex group takes its four colours in two steps: the part of its row
// that reads edge DoFs (44 of 50 terms; unchanged while the colours run) is
// summed once for all colours, with every lane of a warp at work, and each
// colour then adds the few vertex neighbours only.  A colour's sites are
// compact in the lanes (four sites of a row, one of each colour, are one
// slot).  Which site a slot is and which groups have an interior DoF there
// comes from small tables set up once per launch.
//
// A Gauss-Seidel phase only ever updates sites that no site of the same phase
// reads (a vertex colour, or one edge group), so the halo stores of a phase
// never touch values read in that phase.  The same phase twice in a row, at
// the turn of a symmetric sweep, is skipped: with no coupling inside a phase
// its second application reproduces the same values.  The pressure update,
// whose halo stores would reach values the C residual of a neighbour reads,
// follows that residual after a cluster barrier.
//
// Bound: the latency of a phase (barrier, one round of shared loads, the sum,
// the store), on level 4 also the shared-memory loads of 16 CTAs.  Measured
// against the kernel this replaces (rows shared by lanes that walk weight and
// offset tables, every colour with its full row), one forward sweep: P2-P1
// FP32 level 2 / 3 / 4: 8.9 / 11.6 / 21.0 us before, 4.6 / 7.8 / 16.4 us now;
// P1-P1 FP64 level 2 / 3 / 4: 6.2 / 6.9 / 7.6 us before, 3.1 / 3.0 / 4.6 us.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "batch.h"
#include "kernels.h"
#include "small.h"
#include "structure.inc"
#include "weights.h"

namespace cg = cooperative_groups;

namespace hhg {
namespace {

// floor(n / d) for 0 <= n, d < 2^16 from m = floor(2^32 / d) + 1: the
// product n m / 2^32 exceeds n / d by less than n / 2^32 < 1 / d, which never
// reaches the next integer (one wide multiply instead of a division)
__device__ __forceinline__ int qdiv(int n, unsigned long long m) {
  return int((unsigned long long)(unsigned)n * m >> 32);
}
__device__ __forceinline__ unsigned long long qmagic(int d) { return (1ull << 32) / unsigned(d) + 1; }

// sizes of one CTA's shared memory (elements): planes owned at most, planes
// with velocity cells (k < nz) at most
struct ResDims {
  int G, na, pad;          // velocity groups, arrays, odd site stride
  int planes, cells;
  int slab, rhs, np, n, n4, ncb, nw;
};
__host__ __device__ inline int ncb_of(int disc, int varnu) { return disc == 2 ? 0 : varnu ? 15 : 7; }
// compact: the layout of levels that do not fit the other one.  No odd stride,
// no tables of the pressure slots, no edge sums, one thread per pressure row.
__host__ __device__ inline ResDims res_dims(int disc, int varnu, const Geo& g, int C, bool compact) {
  ResDims d;
  d.G = disc == 2 ? 8 : 1;
  d.na = 3 * d.G + 1;
  d.pad = compact ? d.na : d.na | 1;
  d.planes = d.cells = 0;
  for (int c = 0; c < C; ++c) {
    const int kb = int(int64_t(c) * (g.nz + 1) / C), ke = int(int64_t(c + 1) * (g.nz + 1) / C);
    if (ke - kb > d.planes) d.planes = ke - kb;
    const int nc = (ke < g.nz ? ke : g.nz) - kb;
    if (nc > d.cells) d.cells = nc;
  }
  const int sy = int(g.sy);
  d.slab = d.pad * (d.planes + 2) * sy;
  d.np = d.planes * (g.ny + 1) * g.sx;                       // pressure slots (rows padded to the pitch)
  d.n = d.cells * g.ny * g.sx;                               // velocity slots of a component
  d.n4 = d.cells * g.ny * ((g.nx + 3) / 4);                  // vertex slots: four sites of a row
  // right-hand sides of the owned planes (P2: and the edge sums of the
  // vertices), later the partial sums of the pressure row
  const int rhs = (3 * d.G + (disc == 2 && !compact ? 3 : 0)) * d.cells * sy;
  const int parts = (compact ? 1 : disc == 2 ? 3 : 4) * d.np;
  d.rhs = rhs > parts ? rhs : parts;
  d.ncb = ncb_of(disc, varnu);
  d.nw = varnu ? kResMaxTerms : 0;
  return d;
}

// ------------------------------------------------------------- row sums
enum { kAll = 0, kVertex = 1, kEdges = 2 };
// weight of term E of operator table S (index W0 + E in the run-time table;
// constant viscosity: weights.h; W0 = 0: the rows of A)
template <int DISC, class S, int E, int W0, int VARNU, class T>
__device__ __forceinline__ T weight(const T* sw) {
  if constexpr (VARNU) {
    return sw[W0 + E];
  } else {
    constexpr double K = W0 == 0 ? kScaleA<DISC> : kScaleB<DISC>, w = row_weight<S, E, T>(K);
    static_assert(int_weights<S>(E, 1, K), "the scaled weights are small integers");
    return T(w);
  }
}
// adds terms E0 + I that pass the filter: SEL selects vertex or edge inputs,
// COMP >= 0 inputs of that velocity component; p: the site's values; oj, ok:
// the j and k pitch; three chains of sums
template <class S, int E0, int W0, int VARNU, int SEL, int COMP, int G, int PAD, class T, int... I>
__device__ __forceinline__ T row_sum(const T* p, int oj, int ok, const T* sw, std::integer_sequence<int, I...>) {
  T a[3] = {T(0), T(0), T(0)};
  ([&] {
    constexpr gen::OffT o = S::off[E0 + I];
    constexpr bool vertex = o.arr % G == 0;
    if constexpr ((SEL == kAll || (SEL == kVertex) == vertex) && (COMP < 0 || (o.arr < 3 * G && o.arr / G == COMP)))
      a[I % 3] = fma(weight<G == 8 ? 2 : 1, S, E0 + I, W0, VARNU, T>(sw),
                     p[o.arr + PAD * o.di + o.dj * oj + o.dk * ok], a[I % 3]);
  }(), ...);
  return a[0] + a[1] + a[2];
}

// r[g] -= row R0 + g, all of component R0 / G (B^T rows)
template <class S, int R0, int W0, int VARNU, int G, int PAD, class T, int... GG>
__device__ __forceinline__ void bt_rows(T (&r)[G], const T* p, int oj, int ok, const T* sw, const Factor<T>& sb,
                                        std::integer_sequence<int, GG...>) {
  ([&] {
    constexpr gen::RowS rw = S::rows[R0 + GG];
    static_assert(rw.n1 == 0 && rw.n2 == 0, "B^T is unscaled");
    const T s = row_sum<S, rw.t0, W0, VARNU, kAll, -1, G, PAD>(p, oj, ok, sw, std::make_integer_sequence<int, rw.n0>{});
    if constexpr (VARNU != 0) r[GG] -= s;
    else r[GG] = minus_scaled(r[GG], sb, s);
  }(), ...);
}
// the C terms of a pressure row, w: the weights of its boundary class
template <class SPT, int PARR, int PAD, class T, int... O>
__device__ __forceinline__ T c_sum(const T* w, const T* p, int oj, int ok, std::integer_sequence<int, O...>) {
  T s = T(0);
  ((s = fma(w[O], p[PARR + PAD * SPT::cbo[O].di + SPT::cbo[O].dj * oj + SPT::cbo[O].dk * ok], s)), ...);
  return s;
}

// calls f with the value of g in 1 .. 7 as a compile-time constant
template <class F>
__device__ __forceinline__ void with_group(int g, F&& f) {
  switch (g) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    default: f(std::integral_constant<int, 7>{}); break;
  }
}
// calls f with the component of slot q (0 .. 3 n - 1) as a compile-time constant
template <class F>
__device__ __forceinline__ void with_comp(int comp, F&& f) {
  if (comp == 0) f(std::integral_constant<int, 0>{});
  else if (comp == 1) f(std::integral_constant<int, 1>{});
  else f(std::integral_constant<int, 2>{});
}

// the smoother of one cluster (the kernel below, or one work item of a
// merged launch over several problems' clusters)
template <int DISC, int VARNU, bool COMPACT, class T>
__device__ __forceinline__ void uzawa_resident_body(const Geo& g, T* xg, const T* __restrict__ b,
                                                    const double* __restrict__ inv_ml, const SmallArgs& a,
                                                    const ResTabs<T>* __restrict__ tabs, const Factor<T>& sb) {
  using SA = gen::S<DISC, VARNU, OP_A>;
  using SBT = gen::S<DISC, VARNU, OP_BT>;
  using SBC = gen::S<DISC, VARNU, OP_BC>;
  constexpr int G = DISC == 2 ? 8 : 1, NA = 3 * G + 1, PAD = COMPACT ? NA : NA | 1, NPH = 4 + (G - 1);
  constexpr int WBT = SA::N / 3, WBC = WBT + SBT::N;
  static_assert(WBC + SBC::N <= kResMaxTerms, "weights fit the table");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T sdiag[8];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = int(cluster.num_blocks()), c = int(cluster.block_rank());
  const ResDims dm = res_dims(DISC, VARNU, g, C, COMPACT);
  T* xs = reinterpret_cast<T*>(smem_raw);
  T* ts = xs + dm.slab;
  T* mls = ts + dm.rhs;                                      // omega M_L^{-1} of the pressure slots
  T* wc = mls + (COMPACT ? 0 : dm.np);
  T* sw = wc + 27 * dm.ncb;
  int* info = reinterpret_cast<int*>(sw + dm.nw);            // velocity slots: site, groups with an interior DoF
  int* cinfo = info + dm.n;                                  // vertex slots: site of the quad, colour shift
  int* pinfo = cinfo + dm.n4;                                // pressure slots: site, boundary class
  const int nzp = g.nz + 1, nx = g.nx, ny = g.ny;
  const int kb = c * nzp / C, ke = (c + 1) * nzp / C, nk = ke - kb, nc = min(ke, g.nz) - kb;
  const int sx = g.sx, sy = int(g.sy), oj = sx * PAD, ok = sy * PAD;
  const int tid = int(threadIdx.x), nthr = int(blockDim.x);
  // neighbours' slabs: my plane kb is the lower neighbour's upper halo plane,
  // my plane ke-1 the upper neighbour's plane 0
  T* lo = (C > 1 && c > 0) ? cluster.map_shared_rank(xs, c - 1) : nullptr;
  T* hi = (C > 1 && c < C - 1) ? cluster.map_shared_rank(xs, c + 1) : nullptr;
  const int up = c > 0 ? (kb - (c - 1) * nzp / C) * ok : 0, down = nk * ok;
  auto bar = [&] {
    if (C > 1) cluster.sync();
    else __syncthreads();
  };
  auto store = [&](int e, int kl, T v) {           // element of the slab and its halo copies
    xs[e] = v;
    if (kl == 0 && lo) lo[e + up] = v;
    if (kl == nk - 1 && hi) hi[e - down] = v;
  };
  const unsigned long long msy = qmagic(sy), msx = qmagic(sx);
  const int as = dm.cells * sy;                    // stride of the right-hand side arrays
  const int t0 = sy + sx + 1;                      // a site's index in them: its slab site - t0
  // ---- tables and the level's values
  if (tid < G) sdiag[tid] = T(a.inv_diag[tid]);
  for (int q = tid; q < 27 * dm.ncb; q += nthr) wc[q] = tabs->wc[q];
  for (int q = tid; q < dm.nw; q += nthr) sw[q] = tabs->w[q];
  for (int s = tid; s < dm.n; s += nthr) {
    const int row = qdiv(s, msx), i = s - row * sx, kl = row / ny, j = row - kl * ny, k = kb + kl;
    int f = 0;
    if (kl < nc && i < nx)
      for (int gg = 0; gg < G; ++gg) {
        const int ox = (0xB2 >> gg) & 1, oy = (0xD4 >> gg) & 1, oz = (0xE8 >> gg) & 1;
        if ((i > 0 || ox) && (j > 0 || oy) && (k > 0 || oz)) f |= 1 << gg;
      }
    info[s] = ((kl + 1) * sy + (j + 1) * sx + i + 1) | f << 16;
  }
  const int nq = (nx + 3) / 4;
  for (int s = tid; s < dm.n4; s += nthr) {
    const int row = s / nq, i4 = s - row * nq, kl = row / ny, j = row - kl * ny, k = kb + kl;
    cinfo[s] = (kl < nc && j > 0 && k > 0) ? ((kl + 1) * sy + (j + 1) * sx + 1 + 4 * i4) | ((j + k) & 3) << 16 | i4 << 18
                                           : -1;
  }
  auto pslot = [&](int s) {
    const int row = qdiv(s, msx), i = s - row * sx, kl = row / (ny + 1), j = row - kl * (ny + 1), k = kb + kl;
    const int cls = (i == 0 ? 0 : i == nx ? 2 : 1) + 3 * (j == 0 ? 0 : j == ny ? 2 : 1) +
                    9 * (k == 0 ? 0 : k == g.nz ? 2 : 1);
    return kl < nk && i <= nx ? ((kl + 1) * sy + (j + 1) * sx + i + 1) | cls << 16 : -1;
  };
  // omega M_L^{-1} at a slab site
  auto site_ml = [&](int il) { return T(a.inv_omega_inv * inv_ml[int64_t(kb) * sy + il]); };
  if (!COMPACT)
    for (int s = tid; s < dm.np; s += nthr) {
      const int f = pslot(s);
      pinfo[s] = f;
      mls[s] = f < 0 ? T(0) : site_ml(f & 0xffff);
    }
  for (int r = tid; r < (nk + 2) * sy; r += nthr) {          // owned planes and the halo planes kb-1, ke
    T v[NA];
#pragma unroll
    for (int ar = 0; ar < NA; ++ar) v[ar] = xg[ar * g.arr + int64_t(kb) * sy + r];
#pragma unroll
    for (int ar = 0; ar < NA; ++ar) xs[r * PAD + ar] = v[ar];
  }
  bar();                                           // every CTA runs before any remote store

  // (r - s) / diagonal of group row g; constant viscosity: s in the scale of the
  // row's weights, r divided already
  auto over_diag = [&](auto gc, T r, T s) {
    constexpr int GRP = decltype(gc)::value;
    if constexpr (VARNU != 0) {
      return (r - s) * sdiag[GRP];
    } else {
      constexpr Factor<T> f = make_factor<T>(1.0 / row_weight<SA, SA::rows[GRP].t0, T>(kScaleA<DISC>));
      return minus_scaled(r, f, s);
    }
  };
  constexpr std::integral_constant<int, 0> vertex{};
  const int n = dm.n, n3 = 3 * n, m3 = 3 * dm.n4, np = dm.np, nu = (COMPACT ? 1 : DISC == 2 ? 3 : 4) * np;
  constexpr bool kSums = DISC == 2 && !COMPACT;    // the vertex colours share the sums of their edge terms
  for (int it = 0; it < a.iterations; ++it) {
    // ---- velocity step: tmp_u = b_u - B^T p at the interior sites of every group
    for (int q = tid; q < n3; q += nthr) {
      const int comp = (q >= n) + (q >= 2 * n), f = info[q - comp * n], il = f & 0xffff;
      if (!(f >> 16)) continue;
      const T* p = xs + il * PAD;
      const T* bg = b + int64_t(comp * G) * g.arr + int64_t(kb) * sy + il;
      T r[G];
#pragma unroll
      for (int gg = 0; gg < G; ++gg) r[gg] = __ldg(bg + gg * g.arr);
      with_comp(comp, [&](auto cc) {
        constexpr int CO = decltype(cc)::value;
        bt_rows<SBT, CO * G, WBT, VARNU, G, PAD>(r, p, oj, ok, sw, sb,
                                                 std::make_integer_sequence<int, G>{});
      });
      T* t = ts + comp * G * as + il - t0;
#pragma unroll
      for (int gg = 0; gg < G; ++gg) t[gg * as] = r[gg];
    }
    __syncthreads();
    // ---- xi Gauss-Seidel sweeps on A u = tmp_u (forward, and backward for A_s)
    int prev = -1;
    bool sums = false;                             // the vertices' edge sums hold
    for (int sw_ = 0; sw_ < a.xi; ++sw_) {
      for (int pass = 0; pass < (a.ahat == HHG_AHAT_S ? 2 : 1); ++pass) {
        for (int pi = 0; pi < NPH; ++pi) {
          const int ph = pass == 0 ? pi : NPH - 1 - pi;
          if (ph == prev) continue;
          prev = ph;
          if (ph < 4) {
            constexpr gen::RowS rw = SA::rows[0];
            constexpr auto terms = std::make_integer_sequence<int, rw.n1 - 1>{};   // the diagonal is the first term
            if constexpr (kSums) {
              if (!sums) {
                for (int q = tid; q < n3; q += nthr) {
                  const int comp = (q >= n) + (q >= 2 * n), f = info[q - comp * n], il = f & 0xffff;
                  if (!(f >> 16 & 1)) continue;
                  const T s = row_sum<SA, rw.t0 + 1, 0, VARNU, kEdges, -1, G, PAD>(xs + il * PAD + comp * G, oj, ok, sw,
                                                                                   terms);
                  const T r = ts[comp * G * as + il - t0] * (VARNU ? T(g.eisc[kb + qdiv(il, msy) - 1]) : sdiag[0]);
                  ts[(24 + comp) * as + il - t0] = VARNU ? r - s : over_diag(vertex, r, s);
                }
                __syncthreads();
                sums = true;
              }
            }
            for (int q = tid; q < m3; q += nthr) {
              const int comp = (q >= dm.n4) + (q >= 2 * dm.n4), f = cinfo[q - comp * dm.n4];
              const int di = (ph - (f >> 16)) & 3, i = 4 * (f >> 18) + di;
              if (f < 0 || i < 1 || i >= nx) continue;
              const int il = (f & 0xffff) + di, kl = qdiv(il, msy) - 1;
              const T s = row_sum<SA, rw.t0 + 1, 0, VARNU, kSums ? kVertex : kAll, -1, G, PAD>(
                  xs + il * PAD + comp * G, oj, ok, sw, terms);
              T t = ts[(kSums ? 24 + comp : comp * G) * as + il - t0];
              if (!kSums) t *= VARNU ? T(g.eisc[kb + kl]) : sdiag[0];
              store(il * PAD + comp * G, kl, over_diag(vertex, t, s));
            }
          } else if constexpr (DISC == 2) {
            sums = false;
            with_group(ph - 3, [&](auto gc) {
              constexpr int GRP = decltype(gc)::value;
              constexpr gen::RowS rw = SA::rows[GRP];
              const T inv_diag = sdiag[GRP];
              for (int q = tid; q < n3; q += nthr) {
                const int comp = (q >= n) + (q >= 2 * n), f = info[q - comp * n], il = f & 0xffff;
                if (!(f >> (16 + GRP) & 1)) continue;
                const int kl = qdiv(il, msy) - 1;
                const T t = ts[(comp * G + GRP) * as + il - t0];
                const T s = row_sum<SA, rw.t0 + 1, 0, VARNU, kAll, -1, G, PAD>(
                    xs + il * PAD + comp * G, oj, ok, sw, std::make_integer_sequence<int, rw.n1 - 1>{});
                store(il * PAD + comp * G + GRP, kl,
                      over_diag(gc, t * (VARNU ? T(g.eisc[kb + kl]) : inv_diag), s));
              }
            });
          }
          bar();
        }
      }
    }
    // ---- pressure step: tmp_p = g - (B u - C p) at every pressure site, its
    // parts (per velocity component, C) by different threads, then
    // p -= omega M_L^{-1} tmp_p
    auto press_part = [&](int part, int f) {
      const int il = f & 0xffff;
      const T* p = xs + il * PAD;
      T s = T(0);
      if (DISC == 1 && part == 3) {
        using SPT = gen::SP<DISC, VARNU, OP_BC>;
        const T* w = wc + (f >> 16) * SPT::NCB;
        if constexpr (DISC == 1)
          s = c_sum<SPT, 3 * G, PAD>(w, p, oj, ok, std::make_integer_sequence<int, SPT::NCB>{});
        if (VARNU) s *= T(g.eisc[kb + qdiv(il, msy) - 1]);
      } else {
        constexpr gen::RowS rw = SBC::rows[0];
        static_assert(rw.n1 == 0, "B is unscaled");
        with_comp(part, [&](auto cc) {
          s = row_sum<SBC, rw.t0, WBC, VARNU, kAll, decltype(cc)::value, G, PAD>(
              p, oj, ok, sw, std::make_integer_sequence<int, rw.n0>{});
        });
        if (!VARNU) s = scaled(sb, s);
      }
      return s;
    };
    for (int q = tid; q < nu; q += nthr) {
      const int part = COMPACT ? 0 : (q >= np) + (q >= 2 * np) + (q >= 3 * np);
      const int f = COMPACT ? pslot(q) : pinfo[q - part * np];
      if (f < 0) continue;
      if (COMPACT) {
        T v = T(0);
#pragma unroll 1
        for (int c_ = 0; c_ < (DISC == 2 ? 3 : 4); ++c_) v += press_part(c_, f);
        ts[q] = v;
      } else {
        ts[q] = press_part(part, f);
      }
    }
    if (DISC == 1) bar();                          // the neighbours have read the old halo pressures
    else __syncthreads();
    for (int s = tid; s < np; s += nthr) {
      const int f = COMPACT ? pslot(s) : pinfo[s], il = f & 0xffff;
      if (f < 0) continue;
      T v = ts[s];
      if (!COMPACT) v = v + ts[s + np] + ts[s + 2 * np];
      if (DISC == 1 && !COMPACT) v += ts[s + 3 * np];
      const T r = __ldg(b + 3 * G * g.arr + int64_t(kb) * sy + il) - v;
      store(il * PAD + 3 * G, qdiv(il, msy) - 1, xs[il * PAD + 3 * G] - (COMPACT ? site_ml(il) : mls[s]) * r);
    }
    bar();
  }
  // owned planes back to global memory
  for (int r = tid; r < nk * sy; r += nthr) {
#pragma unroll
    for (int ar = 0; ar < NA; ++ar) xg[ar * g.arr + int64_t(kb + 1) * sy + r] = xs[(r + sy) * PAD + ar];
  }
}

template <class T>
struct ResA { Geo g; T* xg; const T* b; const double* inv_ml; SmallArgs a; const ResTabs<T>* tabs; Factor<T> sb; };   // sb: h^2 / K

template <int DISC, int VARNU, bool COMPACT, class T>
__global__ void __launch_bounds__(kResidentThreads, 1) k_uzawa_resident(const __grid_constant__ ResA<T> r) {
  uzawa_resident_body<DISC, VARNU, COMPACT, T>(r.g, r.xg, r.b, r.inv_ml, r.a, r.tabs, r.sb);
}
// every cluster of the merged grid belongs to one item (items start at
// multiples of the cluster size)
template <int DISC, int VARNU, bool COMPACT, class T>
__global__ void __launch_bounds__(kResidentThreads, 1) kb_uzawa_resident(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<ResA<T>>(items, n, bid, gd);
  const ResA<T>& r = it.a;
  uzawa_resident_body<DISC, VARNU, COMPACT, T>(r.g, r.xg, r.b, r.inv_ml, r.a, r.tabs, r.sb);
}

template <class T> constexpr int prec_of() { return sizeof(T) == 8 ? HHG_FP64 : HHG_FP32; }

template <class T>
const void* kernel_of(int disc, int varnu, bool compact, bool batched) {
#define HHG_K(D, V, M)                                                                       \
  if (disc == D && varnu == V && compact == M)                                               \
    return batched ? reinterpret_cast<const void*>(kb_uzawa_resident<D, V, M, T>)            \
                   : reinterpret_cast<const void*>(k_uzawa_resident<D, V, M, T>);
  HHG_K(1, 0, false) HHG_K(1, 1, false) HHG_K(2, 0, false) HHG_K(2, 1, false)
  HHG_K(1, 0, true) HHG_K(1, 1, true) HHG_K(2, 0, true) HHG_K(2, 1, true)
#undef HHG_K
  return nullptr;
}

void fill_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int C, int threads, size_t smem,
                 cudaStream_t s) {
  cfg = {};
  cfg.gridDim = dim3(C, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

}  // namespace

namespace {
size_t layout_smem(int disc, int varnu, const Geo& g, int ctas, int prec, bool compact) {
  const size_t es = prec == HHG_FP64 ? 8 : 4;
  const ResDims d = res_dims(disc, varnu, g, ctas, compact);
  const size_t np = compact ? 0 : d.np;
  return (size_t(d.slab) + d.rhs + np + 27 * d.ncb + d.nw) * es + (size_t(d.n) + d.n4 + np) * 4;
}
}  // namespace

bool resident_compact(int disc, int varnu, const Geo& g, int ctas, int prec) {
  return layout_smem(disc, varnu, g, ctas, prec, false) > kResidentSmemMax;
}
size_t resident_smem(int disc, int varnu, const Geo& g, int ctas, int prec) {
  return layout_smem(disc, varnu, g, ctas, prec, resident_compact(disc, varnu, g, ctas, prec));
}

bool resident_feasible(int disc, int varnu, int prec, const Geo& g, int ctas) {
  if (ctas < 1 || ctas > kResidentMaxCtas || ctas > g.nz + 1) return false;
  // site and slot indices of a CTA stay below 2^16 (qdiv, the packed tables)
  const int64_t planes = (g.nz + 1 + ctas - 1) / ctas + 2;
  if (planes * g.sy >= 65536 || g.nx >= 4 * 8192) return false;
  const size_t smem = resident_smem(disc, varnu, g, ctas, prec);
  if (smem > kResidentSmemMax) return false;
  const bool compact = resident_compact(disc, varnu, g, ctas, prec);
  const void* fn = prec == HHG_FP64 ? kernel_of<double>(disc, varnu, compact, false)
                                    : kernel_of<float>(disc, varnu, compact, false);
  if (!fn || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kResidentSmemMax)) != cudaSuccess ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  fill_config(cfg, attr, ctas, kResidentThreads, smem, nullptr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n > 0;
}

template <class T>
int uzawa_resident(int disc, int varnu, const Geo& g, int ctas, int threads, T* x, const T* b, const double* inv_ml,
                   const SmallArgs& a, const ResTabs<T>* tabs, cudaStream_t s) {
  if (threads < 128 || threads > kResidentThreads || threads % 32) return -1;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  fill_config(cfg, attr, ctas, threads, resident_smem(disc, varnu, g, ctas, prec_of<T>()), s);
  ResA<T> r{g, x, b, inv_ml, a, tabs, make_factor<T>(g.h * g.h / row_scale<T>(disc == 2 ? kScaleB<2> : kScaleB<1>))};
  const bool compact = resident_compact(disc, varnu, g, ctas, prec_of<T>());
  if (g_rec) {
    g_rec->add(kernel_of<T>(disc, varnu, compact, true), dim3(ctas), dim3(threads), cfg.dynamicSmemBytes, ctas, r);
    return 0;
  }
  ++g_launches;
  void* args[] = {&r};
  return cudaLaunchKernelExC(&cfg, kernel_of<T>(disc, varnu, compact, false), args) == cudaSuccess ? 0 : -1;
}

template int uzawa_resident<double>(int, int, const Geo&, int, int, double*, const double*, const double*,
                                    const SmallArgs&, const ResTabs<double>*, cudaStream_t);
template int uzawa_resident<float>(int, int, const Geo&, int, int, float*, const float*, const double*,
                                   const SmallArgs&, const ResTabs<float>*, cudaStream_t);

}  // namespace hhg
