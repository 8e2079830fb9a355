// Refinement residual of the mixed-precision solve in double-float arithmetic.
//
// The mixed solve (FP32 V-cycles inside an FP64 iterative refinement) needs
// the outer residual r = b - calA x of every FMG stage to well below FP32
// rounding.  FP64 arithmetic gives that, but on this GPU FP64 FMAs run at
// about 1/54 of the FP32 rate (1.26 against 68.5 TFLOP/s measured), so the
// FP64 residual of the finest level is bound by them (it was the largest
// single kernel of the level-7 solve).  Here
// every FP64 value v is carried as two FP32 numbers v = v_hi + v_lo (47
// significant bits, split by integer bit operations, no FP64 instruction on
// the common path), and each row is evaluated as the compensated dot product
// "Dot2" of Ogita, Rump and Oishi (Accurate sum and dot product, SIAM J. Sci.
// Comput. 26(6), 2005): the product w_hi x_hi is split exactly into p + e by
// one FMA, p enters the running sum through Knuth's error-free TwoSum (The Art
// of Computer Programming, vol. 2, Sec. 4.2.2), and the sum's rounding errors,
// e and the small products w_lo x_hi + w_hi x_lo are collected in a second
// FP32 accumulator.  With u = 2^-24 and n terms the computed row differs from
// the exact one by at most about u |r| + (n^2 u^2 + 2^-46) sum_j |a_ij x_j|: as
// if evaluated in 47-bit arithmetic and then rounded to FP32, the precision
// the V-cycle takes its right-hand side in.
//
// Work layout.  Constant viscosity but for small levels (k_df_unrolled): a thread owns two sites
// of a plane and a component and applies each (hi, lo) input it loads to all
// the component's rows, two sites per paired FP32 (f32x2) instruction; rows
// are unrolled, with small-integer weights (see there).  Variable viscosity
// and small levels (k_res_df): grid x over the padded (i, j) plane in warps of 4 x 32
// positions, y over groups of kp planes, z over the rows of the operator; on
// large levels a thread evaluates 4 sites 32 positions apart on 2 planes, on
// small ones 1 site on 1 plane, in a loop over weights and offsets in the
// constant bank.
// Boundary pressure rows (P1-P1: the C terms of the cubes inside the box) add
// their per-cube C terms in FP64; they are a few per cent of the pressure
// rows.  With a variable viscosity nu = exp(a z) the segments of a row are
// summed apart and scaled by the row's FP64 factors exp(+-a h k) in
// double-float arithmetic.
#include "dfres.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <utility>

#include "batch.h"
#include "kernels.h"
#include "weights.h"
#include "structure.inc"

namespace hhg {
namespace {

template <int N>
struct DfTab {
  float wh[N];       // weights: w = wh + wl (|w - wh - wl| <= 2^-48 |w|)
  float wl[N];
  int off[N];        // linear offsets arr * array_stride + di + dj sx + dk sy
};

template <int DISC, int VARNU>
using DfTabOf = DfTab<gen::S<DISC, VARNU, OP_FULL>::N>;

// v = hi + lo with |v - hi - lo| < 2^-46 |v|: hi takes the leading 24 bits of
// v's significand, lo the next 23 (both truncated).  For v = 0, |v| < 2^-100
// or |v| >= 2^126, hi = fl32(v) and lo = 0 (an FP64 conversion off the common
// path).
__device__ __forceinline__ void split_df(double v, float& hi, float& lo) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(v));
  const unsigned top = unsigned(u >> 32);
  const unsigned sgn = top & 0x80000000u;
  const int e = int((top >> 20) & 0x7ffu);           // biased FP64 exponent
  if (e >= 923 && e <= 1148) {
    // FP32 exponent field e - 1023 + 127; significand bits 51..29
    hi = __uint_as_float(sgn | (unsigned(e - 896) << 23) | unsigned((u >> 29) & 0x7fffffu));
    // bits 28..6 of the significand scaled by 2^(e - 1069): (1 + f) 2^E - 2^E
    // with E = e - 1046, an exact FP32 subtraction
    const unsigned eb = unsigned(e - 919) << 23;
    lo = __fsub_rn(__uint_as_float(sgn | eb | (unsigned(u & 0x1fffffffu) >> 6)), __uint_as_float(sgn | eb));
  } else if (e == 0) {
    hi = __uint_as_float(sgn);                       // +-0 (and FP64 subnormals, < 2^-1022)
    lo = 0.0f;
  } else {
    hi = __double2float_rn(v);
    lo = 0.0f;
  }
}

// one Dot2 step: (s, c) += (wh + wl) (xh + xl); the rounded operations are
// the _rn intrinsics, which the compiler never contracts into FMAs
__device__ __forceinline__ void dot2_term(float wh, float wl, float xh, float xl, float& s, float& c) {
  const float p = __fmul_rn(wh, xh);
  float e = __fmaf_rn(wh, xh, -p);                   // wh xh = p + e exactly
  e = __fmaf_rn(wl, xh, e);
  e = __fmaf_rn(wh, xl, e);
  const float t = __fadd_rn(s, p);                   // TwoSum: s + p = t + d exactly
  const float z = __fsub_rn(t, s);
  const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(d, e));
}

// a - b on both halves (sub.rn.f32x2: each half rounds as the scalar
// subtraction)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 ra, rb, rr;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " sub.rn.f32x2 rr, ra, rb;\n mov.b64 {%0, %1}, rr;\n}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

// dot2_term on two sites at once with the paired FP32 instructions (each
// half of an f32x2 operation rounds as the scalar one, so the sums are those
// of dot2_term bit for bit)
__device__ __forceinline__ void dot2_term2(float2 wh, float2 wl, float2 xh, float2 xl, float2& s, float2& c) {
  const float2 p = __fmul2_rn(wh, xh);
  float2 e = __ffma2_rn(wh, xh, make_float2(-p.x, -p.y));
  e = __ffma2_rn(wl, xh, e);
  e = __ffma2_rn(wh, xl, e);
  const float2 t = __fadd2_rn(s, p);
  const float2 z = sub2(t, s);
  const float2 d = __fadd2_rn(sub2(s, sub2(t, z)), sub2(p, z));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(d, e));
}

// terms [T0, T0 + N) of a row at NS sites 32 positions apart (idx + 32 v);
// an even NS runs the sites in pairs
template <int T0, int N, int NS, class Tab>
__device__ __forceinline__ void dot2_seg(const Tab& tab, const float* __restrict__ xh, const float* __restrict__ xl,
                                         int64_t idx, float (&s)[NS], float (&c)[NS]) {
  if constexpr (NS % 2 == 0) {
    float2 s2[NS / 2], c2[NS / 2];
#pragma unroll
    for (int h = 0; h < NS / 2; ++h) {
      s2[h] = make_float2(s[2 * h], s[2 * h + 1]);
      c2[h] = make_float2(c[2 * h], c[2 * h + 1]);
    }
#pragma unroll 4
    for (int t = T0; t < T0 + N; ++t) {
      const float wh = tab.wh[t], wl = tab.wl[t];
      const int64_t q = idx + tab.off[t];
#pragma unroll
      for (int h = 0; h < NS / 2; ++h)
        dot2_term2(make_float2(wh, wh), make_float2(wl, wl),
                   make_float2(__ldg(xh + q + 64 * h), __ldg(xh + q + 64 * h + 32)),
                   make_float2(__ldg(xl + q + 64 * h), __ldg(xl + q + 64 * h + 32)), s2[h], c2[h]);
    }
#pragma unroll
    for (int h = 0; h < NS / 2; ++h) {
      s[2 * h] = s2[h].x; s[2 * h + 1] = s2[h].y;
      c[2 * h] = c2[h].x; c[2 * h + 1] = c2[h].y;
    }
  } else {
#pragma unroll 4
    for (int t = T0; t < T0 + N; ++t) {
      const float wh = tab.wh[t], wl = tab.wl[t];
      const int64_t q = idx + tab.off[t];
#pragma unroll
      for (int v = 0; v < NS; ++v) dot2_term(wh, wl, __ldg(xh + q + 32 * v), __ldg(xl + q + 32 * v), s[v], c[v]);
    }
  }
}

// per-cube C terms of boundary pressure row r at site (i, j, k) (index idx),
// the cubes inside the box only, in FP64 with x = xh + xl
__device__ double boundary_c64(const Geo& g, const OpDev& op, int r, int i, int j, int k, const float* xh,
                               const float* xl, int64_t idx) {
  const DRow row = op.rows[r];
  double a = 0.0;
  for (int t = row.b0 + row.m0 + row.m1; t < row.b0 + row.m0 + row.m1 + row.m2; ++t) {
    const DTermB tm = op.bterms[t];
    const int qx = i + tm.cx, qy = j + tm.cy, qz = k + tm.cz;
    if (qx < 0 || qy < 0 || qz < 0 || qx >= g.nx || qy >= g.ny || qz >= g.nz) continue;
    const int64_t q = int64_t(tm.arr) * g.arr + idx + tm.off;
    a += __ldg(op.bw64 + t) * (double(__ldg(xh + q)) + double(__ldg(xl + q)));
  }
  return a;
}

// (s, c) += a (u + v) for an FP64 factor a = ah + al: ah u = p + e exactly
// (FMA), the small products into e, p into the sum by TwoSum
__device__ __forceinline__ void df_add_scaled(double a, float u, float v, float& s, float& c) {
  float ah, al;
  split_df(a, ah, al);
  const float p = __fmul_rn(ah, u);
  float e = __fmaf_rn(ah, u, -p);
  e = __fmaf_rn(ah, v, e);
  e = __fmaf_rn(al, u, e);
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(d, e));
}

// the residual of row R at one site from its sums: (s, c) over segment 0
// (and segment 1 with a constant viscosity), (s1, c1) over segment 1 with a
// variable one (scaled by exp(+nu_a h k)), (s2, c2) over segment 2 (C; scaled
// by exp(-nu_a h k) with a variable viscosity); bnd: the site lies on the box
// boundary
template <int OUT, int ALL, int N2, int VARNU>
__device__ __forceinline__ void df_store(const Geo& g, const OpDev& op, int R, int i, int j, int k, bool bnd,
                                         const float* xh, const float* xl, int64_t idx, float s, float c, float s1,
                                         float c1, float s2, float c2, const double* __restrict__ b,
                                         float* __restrict__ r) {
  const int64_t iy = int64_t(OUT) * g.arr + idx;
  if (bnd && !ALL) {                                 // Dirichlet velocity row
    r[iy] = 0.0f;
    return;
  }
  const double bv = __ldg(b + iy);
  const double es = VARNU ? __ldg(g.esc + k) : 1.0, eis = VARNU ? __ldg(g.eisc + k) : 1.0;
  if (N2 > 0 && bnd) {
    // boundary pressure row: the clipped C terms in FP64
    const double cb = boundary_c64(g, op, R, i, j, k, xh, xl, idx);
    const double a1 = VARNU ? es * (double(s1) + double(c1)) : 0.0;
    r[iy] = __double2float_rn(bv - (double(s) + double(c)) - a1 - eis * cb);
    return;
  }
  if (VARNU) {
    df_add_scaled(es, s1, c1, s, c);
    if (N2 > 0) df_add_scaled(eis, s2, c2, s, c);
  } else if (N2 > 0) {                               // (s, c) += (s2, c2)
    const float t = __fadd_rn(s, s2);
    const float z = __fsub_rn(t, s);
    const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(s2, z));
    s = t;
    c = __fadd_rn(c, __fadd_rn(c2, d));
  }
  float bh, bl;
  split_df(bv, bh, bl);
  // (bh + bl) - (s + c): TwoSum of bh and -s, then the small parts
  const float t = __fsub_rn(bh, s);
  const float z = __fsub_rn(t, bh);
  const float d = __fadd_rn(__fsub_rn(bh, __fsub_rn(t, z)), __fsub_rn(-s, z));
  r[iy] = __fadd_rn(t, __fsub_rn(__fadd_rn(d, bl), c));
}

// row R = (OUT, OG, ALL, T0, N0, N1, N2) on the sites of the block: the
// indexing in the file's header (V runs of 32 positions per warp; a
// warp whose last run passes the group's last site takes its sites one by one)
template <int V, int VARNU, int OUT, int OG, int ALL, int T0, int N0, int N1, int N2, class Tab>
__device__ __forceinline__ void df_rows(const uint3 bid, const Geo& g, int R, const float* __restrict__ xh,
                                        const float* __restrict__ xl, const double* __restrict__ b,
                                        float* __restrict__ r, const OpDev& op, const Tab& tab, int kp) {
  constexpr int ox = OG == 1 || OG == 4 || OG == 5 || OG == 7;
  constexpr int oy = OG == 2 || OG == 4 || OG == 6 || OG == 7;
  constexpr int oz = OG == 3 || OG == 5 || OG == 6 || OG == 7;
  const int m0 = ((bid.x * blockDim.x + threadIdx.x) >> 5) * (32 * V);
  const int lane = int(threadIdx.x & 31);
  const int mlast = (g.ny - oy) * g.sx + (g.nx - ox);
  if (m0 > mlast) return;
  const int k0 = bid.y * kp, k1 = min(k0 + kp, g.nz - oz + 1);
  if (m0 + 32 * V - 1 > mlast) {                     // warp-uniform: the plane's last warp
#pragma unroll 1
    for (int k = k0; k < k1; ++k)
#pragma unroll 1
      for (int v = 0; v < V; ++v) {
        const int m = m0 + lane + 32 * v;
        const int j = m / g.sx, i = m - j * g.sx;
        if (m > mlast || i > g.nx - ox) continue;
        const bool bnd = 2 * i + ox == 0 || 2 * i + ox == 2 * g.nx || 2 * j + oy == 0 || 2 * j + oy == 2 * g.ny ||
                         2 * k + oz == 0 || 2 * k + oz == 2 * g.nz;
        const int64_t idx = int64_t(m) + 1 + g.sx + int64_t(k + 1) * g.sy;
        float s[1] = {0.0f}, c[1] = {0.0f}, s1[1] = {0.0f}, c1[1] = {0.0f}, s2[1] = {0.0f}, c2[1] = {0.0f};
        if (!bnd || ALL) {
          if (VARNU) {
            dot2_seg<T0, N0, 1>(tab, xh, xl, idx, s, c);
            dot2_seg<T0 + N0, N1, 1>(tab, xh, xl, idx, s1, c1);
          } else {
            dot2_seg<T0, N0 + N1, 1>(tab, xh, xl, idx, s, c);
          }
          if (N2 > 0 && !bnd) dot2_seg<T0 + N0 + N1, N2, 1>(tab, xh, xl, idx, s2, c2);
        }
        df_store<OUT, ALL, N2, VARNU>(g, op, R, i, j, k, bnd, xh, xl, idx, s[0], c[0], s1[0], c1[0], s2[0], c2[0], b,
                                      r);
      }
    return;
  }
  int iv[V], jv[V];
  bool okv[V], bijv[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int m = m0 + lane + 32 * v;
    jv[v] = m / g.sx;
    iv[v] = m - jv[v] * g.sx;
    okv[v] = iv[v] <= g.nx - ox;
    bijv[v] = 2 * iv[v] + ox == 0 || 2 * iv[v] + ox == 2 * g.nx || 2 * jv[v] + oy == 0 || 2 * jv[v] + oy == 2 * g.ny;
  }
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const int64_t idx = int64_t(m0 + lane) + 1 + g.sx + int64_t(k + 1) * g.sy;
    float s[V], c[V], s1[V], c1[V], s2[V], c2[V];
#pragma unroll
    for (int v = 0; v < V; ++v) s[v] = c[v] = s1[v] = c1[v] = s2[v] = c2[v] = 0.0f;
    if (VARNU) {
      dot2_seg<T0, N0, V>(tab, xh, xl, idx, s, c);
      dot2_seg<T0 + N0, N1, V>(tab, xh, xl, idx, s1, c1);
    } else {
      dot2_seg<T0, N0 + N1, V>(tab, xh, xl, idx, s, c);
    }
    if (N2 > 0) dot2_seg<T0 + N0 + N1, N2, V>(tab, xh, xl, idx, s2, c2);
    const bool bk = 2 * k + oz == 0 || 2 * k + oz == 2 * g.nz;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (okv[v])
        df_store<OUT, ALL, N2, VARNU>(g, op, R, iv[v], jv[v], k, bijv[v] || bk, xh, xl, idx + 32 * v, s[v], c[v],
                                      s1[v], c1[v], s2[v], c2[v], b, r);
  }
}

template <class S, int R, class F>
__device__ __forceinline__ void by_row(int r, F&& f) {
  if constexpr (R < S::R) {
    if (r == R) f(std::integral_constant<int, R>{});
    else by_row<S, R + 1>(r, f);
  }
}

template <int DISC, int VARNU, int V, class Tab>
__device__ __forceinline__ void res_df_body(const uint3 bid, const Geo& g, const float* __restrict__ xh,
                                            const float* __restrict__ xl, const double* __restrict__ b,
                                            float* __restrict__ r, const OpDev& op, int kp, const Tab& tab) {
  using S = gen::S<DISC, VARNU, OP_FULL>;
  by_row<S, 0>(int(bid.z), [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    constexpr gen::RowS rw = S::rows[R];
    df_rows<V, VARNU, rw.out, rw.og, rw.all, rw.t0, rw.n0, rw.n1, rw.n2>(bid, g, R, xh, xl, b, r, op, tab, kp);
  });
}

template <int DISC, int VARNU, int V>
__global__ void __launch_bounds__(128) k_res_df(Geo g, const float* __restrict__ xh, const float* __restrict__ xl,
                                                const double* __restrict__ b, float* __restrict__ r, OpDev op, int kp,
                                                const __grid_constant__ DfTabOf<DISC, VARNU> tab) {
  res_df_body<DISC, VARNU, V>(blockIdx, g, xh, xl, b, r, op, kp, tab);
}

// ---------------------------------------------- constant viscosity, unrolled
// With a constant viscosity the weights at h = 1 are multiples of 1 / 15 (A)
// and 1 / 60 (B, B^T; P1-P1: 1 and 1 / 12): times K = 15, 60 (1, 12) they are
// small integers, exact in FP32, so a term has no low weight part, and a term
// whose integer is a power of two has an exact product.  A row then takes the
// factor h / K (h^2 / K) once, in double-float arithmetic.  Only the interior
// C terms of P1-P1 (weights with |T|^(2/3)) keep two-part weights.  Eight to
// eleven operations per term instead of twelve, two loads per input instead of
// per term, no loop: the loop over table entries that this replaces spent about
// 20 instructions per term and site.  P2-P1 level 7, with the split of x: 1.75
// ms before, 1.15 ms now; level 6: 259 us before, 171 us.  Bound: instruction
// issue.
constexpr bool power_of_two(double v) {
  if (v < 0) v = -v;
  for (double p = 1.0; p <= 64.0; p *= 2.0)
    if (v == p) return true;
  return false;
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

// (s, c) += p + e on two sites: TwoSum of s and p
__device__ __forceinline__ void add_exact2(float2 p, float2 e, float2& s, float2& c) {
  const float2 t = __fadd2_rn(s, p);
  const float2 z = sub2(t, s);
  const float2 d = __fadd2_rn(sub2(s, sub2(t, z)), sub2(p, z));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(d, e));
}

// term E of operator table S times K: the integer weight (or, K = 0, the
// two-part weight at h = 1) times x on two sites
template <class S, int E, int K>
__device__ __forceinline__ void unrolled_term(float2 xh, float2 xl, float2& s, float2& c) {
  if constexpr (K == 0) {
    constexpr double w = S::wref[E];
    constexpr float wh = float(w), wl = float(w - double(wh));
    dot2_term2(both(wh), both(wl), xh, xl, s, c);
  } else {
    constexpr double wk = S::wref[E] * K;
    static_assert(near_integer(wk) && wk > -1024.0 && wk < 1024.0, "the scaled weights are small integers");
    constexpr float w = float(rounded(wk));
    if constexpr (power_of_two(w)) {
      add_exact2(__fmul2_rn(both(w), xh), __fmul2_rn(both(w), xl), s, c);
    } else {
      const float2 p = __fmul2_rn(both(w), xh);
      add_exact2(p, __ffma2_rn(both(w), xl, __ffma2_rn(both(w), xh, neg2(p))), s, c);
    }
  }
}

// (s, c) = a (s + c) for an FP64 factor a
__device__ __forceinline__ void df_scale(double a, float& s, float& c) {
  float u = s, v = c;
  s = c = 0.0f;
  df_add_scaled(a, u, v, s, c);
}

// two sites of the split vector: d positions apart
struct Pair {
  const float* h0; const float* h1; const float* l0; const float* l1;
  __device__ __forceinline__ float2 hi(int64_t o) const { return make_float2(__ldg(h0 + o), __ldg(h1 + o)); }
  __device__ __forceinline__ float2 lo(int64_t o) const { return make_float2(__ldg(l0 + o), __ldg(l1 + o)); }
};

// the terms of line L of the full operator's plan at i offset DI, pressure
// inputs (PR) or velocity inputs, on the pass's velocity rows
template <class S, class SPT, int Q, int L, int DI, int K>
constexpr bool df_line_reads() {
  for (int e = SPT::lines[L].e0; e < SPT::lines[L].e0 + SPT::lines[L].ne; ++e)
    if (SPT::terms[e].di == DI && !SPT::parts[SPT::passes[Q].p0 + SPT::terms[e].part].all) return true;
  return false;
}
template <class S, class SPT, int Q, int L, int DI, int K, int NP, int... I>
__device__ __forceinline__ void df_line_value(const Pair& p, int64_t o, float2 (&s)[NP], float2 (&c)[NP],
                                              std::integer_sequence<int, I...>) {
  if constexpr (df_line_reads<S, SPT, Q, L, DI, K>()) {
    const float2 xh = p.hi(o + DI), xl = p.lo(o + DI);
    ([&] {
      constexpr gen::TermE te = SPT::terms[SPT::lines[L].e0 + I];
      if constexpr (te.di == DI && !SPT::parts[SPT::passes[Q].p0 + te.part].all)
        unrolled_term<S, te.t, K>(xh, xl, s[te.part], c[te.part]);
    }(), ...);
  }
}
template <class S, class SPT, int Q, int L, int PARR, bool PR, int K, int NP>
__device__ __forceinline__ void df_line(const Geo& g, const Pair& p, float2 (&s)[NP], float2 (&c)[NP]) {
  constexpr gen::LineT ln = SPT::lines[L];
  constexpr int arr = SPT::arrs[SPT::passes[Q].a0 + ln.slot];
  if constexpr ((arr == PARR) == PR) {
    const int64_t o = arr * g.arr + ln.dj * g.sx + ln.dk * g.sy;
    const auto all = std::make_integer_sequence<int, ln.ne>{};
    df_line_value<S, SPT, Q, L, -1, K>(p, o, s, c, all);
    df_line_value<S, SPT, Q, L, 0, K>(p, o, s, c, all);
    df_line_value<S, SPT, Q, L, 1, K>(p, o, s, c, all);
  }
}
template <class S, class SPT, int Q, int PARR, bool PR, int K, int NP, int... L>
__device__ __forceinline__ void df_lines(const Geo& g, const Pair& p, float2 (&s)[NP], float2 (&c)[NP],
                                         std::integer_sequence<int, L...>) {
  (df_line<S, SPT, Q, SPT::passes[Q].l0 + L, PARR, PR, K>(g, p, s, c), ...);
}
// terms [T0, T0 + n) of a row in two chains, added up
template <class S, int T0, int K, int... I>
__device__ __forceinline__ void df_chain(const Geo& g, const Pair& p, float2& s, float2& c,
                                         std::integer_sequence<int, I...>) {
  float2 s2[3] = {}, c2[3] = {};
  ([&] {
    constexpr gen::OffT o = S::off[T0 + I];
    const int64_t q = o.arr * g.arr + o.di + o.dj * g.sx + o.dk * g.sy;
    unrolled_term<S, T0 + I, K>(p.hi(q), p.lo(q), s2[I % 3], c2[I % 3]);
  }(), ...);
  s = s2[0];
  c = c2[0];
  add_exact2(s2[1], c2[1], s, c);
  add_exact2(s2[2], c2[2], s, c);
}

struct DfA { Geo g; const float* xh; const float* xl; const double* b; float* r; OpDev op; int d; };

// the rows of pass Q (P2-P1: a component, P1-P1: all three) at two sites
template <int DISC, int Q, int... P>
__device__ __forceinline__ void df_velocity(const DfA& a, const Pair& p, const int (&i)[2], const int (&j)[2], int k,
                                            const int64_t (&idx)[2], std::integer_sequence<int, P...>) {
  using S = gen::S<DISC, 0, OP_FULL>;
  using SPT = gen::SP<DISC, 0, OP_FULL>;
  constexpr gen::PassT ps = SPT::passes[Q];
  constexpr int PARR = DISC == 2 ? 24 : 3;
  const Geo& g = a.g;
  float2 s[ps.np] = {}, c[ps.np] = {};
  const auto lines = std::make_integer_sequence<int, ps.nl>{};
  // B^T first, brought to the scale of A: (h^2 / KB) / (h / KA)
  df_lines<S, SPT, Q, PARR, true, int(kScaleB<DISC>)>(g, p, s, c, lines);
  const double ratio = g.h * (kScaleA<DISC> / kScaleB<DISC>);
#pragma unroll
  for (int r = 0; r < ps.np; ++r) {
    df_scale(ratio, s[r].x, c[r].x);
    df_scale(ratio, s[r].y, c[r].y);
  }
  df_lines<S, SPT, Q, PARR, false, int(kScaleA<DISC>)>(g, p, s, c, lines);
  const double scale = g.h / kScaleA<DISC>;
  ([&] {
    constexpr gen::PartT pt = SPT::parts[ps.p0 + P];
    if constexpr (!pt.all) {
      constexpr int ox = (0xB2 >> pt.og) & 1, oy = (0xD4 >> pt.og) & 1, oz = (0xE8 >> pt.og) & 1;
      df_scale(scale, s[P].x, c[P].x);
      df_scale(scale, s[P].y, c[P].y);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        if (i[v] > g.nx - ox || j[v] > g.ny - oy || k > g.nz - oz) continue;
        const bool bnd = (!ox && (i[v] == 0 || i[v] == g.nx)) || (!oy && (j[v] == 0 || j[v] == g.ny)) ||
                         (!oz && (k == 0 || k == g.nz));
        df_store<pt.out, 0, 0, 0>(g, a.op, pt.row, i[v], j[v], k, bnd, a.xh, a.xl, idx[v], v ? s[P].y : s[P].x,
                                  v ? c[P].y : c[P].x, 0.0f, 0.0f, 0.0f, 0.0f, a.b, a.r);
      }
    }
  }(), ...);
}
template <int DISC>
__device__ __forceinline__ void df_pressure(const DfA& a, const Pair& p, const int (&i)[2], const int (&j)[2], int k,
                                            const int64_t (&idx)[2]) {
  using S = gen::S<DISC, 0, OP_FULL>;
  constexpr int PARR = DISC == 2 ? 24 : 3;
  constexpr gen::RowS rw = S::rows[PARR];
  static_assert(rw.out == PARR && rw.n1 == 0, "the last row is the pressure's; B is unscaled");
  const Geo& g = a.g;
  float2 s, c, s2 = {}, c2 = {};
  df_chain<S, rw.t0, int(kScaleB<DISC>)>(g, p, s, c, std::make_integer_sequence<int, rw.n0>{});
  const double sb = g.h * g.h / kScaleB<DISC>;
  df_scale(sb, s.x, c.x);
  df_scale(sb, s.y, c.y);
  if constexpr (rw.n2 > 0) {
    df_chain<S, rw.t0 + rw.n0, 0>(g, p, s2, c2, std::make_integer_sequence<int, rw.n2>{});
    const double sc = g.h * g.h * g.h;
    df_scale(sc, s2.x, c2.x);
    df_scale(sc, s2.y, c2.y);
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    if (i[v] > g.nx || j[v] > g.ny) continue;
    const bool bnd = i[v] == 0 || i[v] == g.nx || j[v] == 0 || j[v] == g.ny || k == 0 || k == g.nz;
    df_store<PARR, 1, rw.n2, 0>(g, a.op, PARR, i[v], j[v], k, bnd, a.xh, a.xl, idx[v], v ? s.y : s.x, v ? c.y : c.x,
                                0.0f, 0.0f, v ? s2.y : s2.x, v ? c2.y : c2.x, a.b, a.r);
  }
}

// grid x over the positions m = i + j sx of the padded (i, j) plane in warps
// of 64 (a lane's two sites lie d = 32 apart; the last warp starts early
// enough to end with the plane's last site, and planes of less than 64
// positions take one site per lane: d = 0), y = plane, z = part: the
// components (P1-P1: all at once), then the pressure
template <int DISC>
__device__ __forceinline__ void df_unrolled_body(const uint3 bid, const DfA& a) {
  using SPT = gen::SP<DISC, 0, OP_FULL>;
  const Geo& g = a.g;
  const int mlast = g.ny * g.sx + g.nx, span = a.d ? 64 : 32, lane = int(threadIdx.x & 31);
  int m0 = int((bid.x * blockDim.x + threadIdx.x) >> 5) * span;
  if (m0 > mlast) return;
  if (a.d) m0 = min(m0, mlast - 63);
  const int k = bid.y;
  int i[2], j[2];
  int64_t idx[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int m = min(m0 + lane + v * a.d, mlast);
    j[v] = m / g.sx;
    i[v] = m - j[v] * g.sx;
    idx[v] = int64_t(m) + 1 + g.sx + int64_t(k + 1) * g.sy;
  }
  const Pair p{a.xh + idx[0], a.xh + idx[1], a.xl + idx[0], a.xl + idx[1]};
  if constexpr (DISC == 1) {
    if (bid.z == 0) df_velocity<1, 0>(a, p, i, j, k, idx, std::make_integer_sequence<int, SPT::passes[0].np>{});
    else df_pressure<1>(a, p, i, j, k, idx);
  } else {
    if (bid.z == 0) df_velocity<2, 0>(a, p, i, j, k, idx, std::make_integer_sequence<int, SPT::passes[0].np>{});
    else if (bid.z == 1) df_velocity<2, 1>(a, p, i, j, k, idx, std::make_integer_sequence<int, SPT::passes[1].np>{});
    else if (bid.z == 2) df_velocity<2, 2>(a, p, i, j, k, idx, std::make_integer_sequence<int, SPT::passes[2].np>{});
    else df_pressure<2>(a, p, i, j, k, idx);
  }
}
template <int DISC>
__global__ void __launch_bounds__(128) k_df_unrolled(const __grid_constant__ DfA a) {
  df_unrolled_body<DISC>(blockIdx, a);
}
template <int DISC>
__global__ void __launch_bounds__(128) kb_df_unrolled(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<DfA>(items, n, bid, gd);
  df_unrolled_body<DISC>(bid, it.a);
}

// hi[q] + lo[q] = x[q] (split_df), two elements per thread and step (n even)
__device__ __forceinline__ void split_df_body(const uint3 bid, const uint3 gd, const double2* __restrict__ x,
                                              float2* __restrict__ hi, float2* __restrict__ lo, int64_t n2) {
  for (int64_t q = bid.x * int64_t(blockDim.x) + threadIdx.x; q < n2; q += int64_t(gd.x) * blockDim.x) {
    const double2 v = x[q];
    float2 h, l;
    split_df(v.x, h.x, l.x);
    split_df(v.y, h.y, l.y);
    hi[q] = h;
    lo[q] = l;
  }
}

__global__ void k_split_df(const double2* __restrict__ x, float2* __restrict__ hi, float2* __restrict__ lo,
                           int64_t n2) {
  split_df_body(blockIdx, gridDim, x, hi, lo, n2);
}

// the same two kernels as work items of a merged batch launch (batch.h; the
// weight table as a device copy)
struct SplitA { const double2* x; float2* hi; float2* lo; int64_t n2; };
template <class Tab>
struct ResDfA { Geo g; const float* xh; const float* xl; const double* b; float* r; OpDev op; int kp; const Tab* tab; };

__global__ void kb_split_df(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<SplitA>(items, n, bid, gd);
  split_df_body(bid, gd, it.a.x, it.a.hi, it.a.lo, it.a.n2);
}

template <int DISC, int VARNU, int V>
__global__ void __launch_bounds__(128) kb_res_df(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<ResDfA<DfTabOf<DISC, VARNU>>>(items, n, bid, gd);
  const auto& a = it.a;
  res_df_body<DISC, VARNU, V>(bid, a.g, a.xh, a.xl, a.b, a.r, a.op, a.kp, *a.tab);
}

constexpr int kDfThreads = 128;
// levels with at most this many lattice sites take one site and one plane
// per thread (the row loops are latency-bound; more threads hide it), larger
// ones four sites and two planes
constexpr int64_t kDfSmallSites = 300000;
// constant viscosity: levels with at most this many sites run the looped
// kernel too.  They are bound by the fetch of code that each warp runs once,
// and the loop is short: defect of P2-P1 with 729 sites 18.5 us looped, 22.6
// us unrolled; 4913 sites 24.7 and 22.6 us; P1-P1 with 35937 sites 26.7 and
// 30.8 us; 105633 sites 35.2 and 30.8 us.
template <int DISC>
constexpr int64_t kDfLoopSites = DISC == 2 ? 4000 : 60000;

template <int DISC>
void launch_df_unrolled(const Geo& g, const OpDev& od, const double* x, const double* b, float* xh, float* xl,
                        float* r, cudaStream_t s) {
  const int64_t n2 = (3 * int64_t(g.G) + 1) * g.arr / 2;   // arr is a multiple of 64
  const dim3 sgrd(unsigned(std::min<int64_t>((n2 + 255) / 256, 152 * 8)));
  const SplitA sa{reinterpret_cast<const double2*>(x), reinterpret_cast<float2*>(xh), reinterpret_cast<float2*>(xl),
                  n2};
  const int mlast = g.ny * g.sx + g.nx, span = mlast >= 63 ? 64 : 32;
  const int warps = mlast / span + 1;
  const dim3 grd(unsigned((warps * 32 + kDfThreads - 1) / kDfThreads), unsigned(g.nz + 1), DISC == 2 ? 4 : 2);
  const DfA a{g, xh, xl, b, r, od, mlast >= 63 ? 32 : 0};
  if (g_rec) {
    g_rec->add(reinterpret_cast<const void*>(kb_split_df), sgrd, dim3(256), 0, 1, sa);
    g_rec->add(reinterpret_cast<const void*>(kb_df_unrolled<DISC>), grd, dim3(kDfThreads), 0, 1, a);
    return;
  }
  ++g_launches;
  k_split_df<<<sgrd, 256, 0, s>>>(sa.x, sa.hi, sa.lo, n2);
  ++g_launches;
  k_df_unrolled<DISC><<<grd, kDfThreads, 0, s>>>(a);
}

template <int DISC, int VARNU>
void launch_df(const Geo& g, const OpDev& od, const char* tab, const double* x, const double* b, float* xh, float* xl,
               float* r, cudaStream_t s) {
  using S = gen::S<DISC, VARNU, OP_FULL>;
  using Tab = DfTabOf<DISC, VARNU>;
  const int64_t n = (3 * int64_t(g.G) + 1) * g.arr;  // a multiple of 64
  const int64_t n2 = n / 2;
  const dim3 sgrd(unsigned(std::min<int64_t>((n2 + 255) / 256, 152 * 8)));
  const SplitA sa{reinterpret_cast<const double2*>(x), reinterpret_cast<float2*>(xh), reinterpret_cast<float2*>(xl),
                  n2};
  const bool small = VARNU == 0 || int64_t(g.nx + 1) * (g.ny + 1) * (g.nz + 1) <= kDfSmallSites;
  const int v = small ? 1 : 4, kp = small ? 1 : 2;
  // warps of v x 32 positions over the padded plane up to the last site
  const int64_t warps = ((int64_t(g.ny) * g.sx + g.nx + 1) + 32 * v - 1) / (32 * v);
  const dim3 grd(unsigned((warps * 32 + kDfThreads - 1) / kDfThreads), unsigned((g.nz + 1 + kp - 1) / kp),
                 unsigned(S::R));
  if (g_rec) {                                       // a batch records: two work items
    const Tab* dt = static_cast<const Tab*>(g_rec->table(tab, sizeof(Tab)));
    g_rec->add(reinterpret_cast<const void*>(kb_split_df), sgrd, dim3(256), 0, 1, sa);
    g_rec->add(small ? reinterpret_cast<const void*>(kb_res_df<DISC, VARNU, 1>)
                     : reinterpret_cast<const void*>(kb_res_df<DISC, VARNU, VARNU ? 4 : 1>),
               grd, dim3(kDfThreads), 0, 1, ResDfA<Tab>{g, xh, xl, b, r, od, kp, dt});
    return;
  }
  Tab tb;
  std::memcpy(&tb, tab, sizeof(tb));
  ++g_launches;
  k_split_df<<<sgrd, 256, 0, s>>>(sa.x, sa.hi, sa.lo, n2);
  ++g_launches;
  if (small) k_res_df<DISC, VARNU, 1><<<grd, kDfThreads, 0, s>>>(g, xh, xl, b, r, od, kp, tb);
  else k_res_df<DISC, VARNU, VARNU ? 4 : 1><<<grd, kDfThreads, 0, s>>>(g, xh, xl, b, r, od, kp, tb);
}

void df_launch(int disc, int varnu, const Geo& g, const OpDev& od, const char* tab, const double* x, const double* b,
               float* xh, float* xl, float* r, cudaStream_t s) {
  const int64_t sites = int64_t(g.nx + 1) * (g.ny + 1) * (g.nz + 1);
  if (disc == 1 && !varnu && sites <= kDfLoopSites<1>) launch_df<1, 0>(g, od, tab, x, b, xh, xl, r, s);
  else if (disc == 2 && !varnu && sites <= kDfLoopSites<2>) launch_df<2, 0>(g, od, tab, x, b, xh, xl, r, s);
  else if (disc == 1 && !varnu) launch_df_unrolled<1>(g, od, x, b, xh, xl, r, s);
  else if (disc == 1) launch_df<1, 1>(g, od, tab, x, b, xh, xl, r, s);
  else if (!varnu) launch_df_unrolled<2>(g, od, x, b, xh, xl, r, s);
  else launch_df<2, 1>(g, od, tab, x, b, xh, xl, r, s);
}

}  // namespace

bool df_supported(int disc, int varnu) { return (varnu == 0 || varnu == 1) && (disc == 1 || disc == 2); }

bool df_table(int disc, int varnu, const std::vector<char>& ftab64, std::vector<char>& out) {
  out.clear();
  if (!df_supported(disc, varnu)) return false;
  const int N = disc == 1 ? (varnu ? gen::S<1, 1, OP_FULL>::N : gen::S<1, 0, OP_FULL>::N)
                          : (varnu ? gen::S<2, 1, OP_FULL>::N : gen::S<2, 0, OP_FULL>::N);
  const size_t bytes = disc == 1 ? (varnu ? sizeof(DfTabOf<1, 1>) : sizeof(DfTabOf<1, 0>))
                                 : (varnu ? sizeof(DfTabOf<2, 1>) : sizeof(DfTabOf<2, 0>));
  if (ftab64.size() < size_t(N) * 12) return false;
  // the FP64 table image: N weights, then N offsets
  const double* w = reinterpret_cast<const double*>(ftab64.data());
  const int* off = reinterpret_cast<const int*>(ftab64.data() + size_t(N) * 8);
  out.assign(bytes, 0);
  float* wh = reinterpret_cast<float*>(out.data());
  float* wl = wh + N;
  int* o = reinterpret_cast<int*>(out.data() + size_t(2 * N) * 4);
  for (int t = 0; t < N; ++t) {
    wh[t] = float(w[t]);
    wl[t] = float(w[t] - double(wh[t]));
    o[t] = off[t];
  }
  return true;
}

void df_residual(int disc, int varnu, const Geo& g, const OpDev& od, const std::vector<char>& dftab, const double* x,
                 const double* b, float* xh, float* xl, float* r, cudaStream_t s) {
  df_launch(disc, varnu, g, od, dftab.data(), x, b, xh, xl, r, s);
}

}  // namespace hhg
