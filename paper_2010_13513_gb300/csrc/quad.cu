// B^T and the pressure step of the Uzawa smoother, P1-P1 in FP32, on large
// levels.
//
// A thread owns four consecutive sites, 16-byte aligned, of a plane: of each
// line its rows read (seven neighbouring lines of an array) it loads four
// values at once, takes the value before and after them from its neighbours in
// the warp (lanes 0 and 31 load theirs), and applies them to every term that
// reads them.  Blocks march over four planes, so that the lines of
// neighbouring rows and planes meet in L1.  Weights come from the constant
// bank.  Boundary pressure rows keep the merged B terms (exact for inputs with
// zero Dirichlet velocities) and take the C stencil of their boundary class.
//
// Bound: load latency, with HBM next (17 million sites, variable viscosity:
// B^T 132 us, pressure step 270 us; their vectors once over HBM 72 and 83 us).
// The same scheme for the whole operator was slower than the streaming
// kernels (311 us against 230 us).
#include "quad.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <utility>

#include "at.h"
#include "batch.h"
#include "structure.inc"

namespace hhg {
namespace {

struct QuadA {
  Geo g; const float* x; const float* b; float* y; const ResTabs<float>* tabs; const double* inv_ml; double s; int kp;
};
template <int VARNU, int OP>
struct QuadTab { float w[gen::S<1, VARNU, OP>::N]; };

__device__ __forceinline__ float4 ld4(const float* base, unsigned off) {
  return __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const char*>(base) + off));
}

// whether line L has a term at i offset DI
template <class SPT, int L, int DI>
constexpr bool quad_reads() {
  for (int e = SPT::lines[L].e0; e < SPT::lines[L].e0 + SPT::lines[L].ne; ++e)
    if (SPT::terms[e].di == DI) return true;
  return false;
}
// the terms of line L at the thread's four sites: acc[part][B / B^T or A, C][site]
template <class SPT, int L, int NP, class Tab, int... I>
__device__ __forceinline__ void quad_line(const Geo& g, const float* __restrict__ x, const Lines<float>& at, bool lo,
                                          bool hi, const Tab& tab, float (&acc)[NP][2][4],
                                          std::integer_sequence<int, I...>) {
  constexpr gen::LineT ln = SPT::lines[L];
  constexpr int arr = SPT::arrs[SPT::passes[0].a0 + ln.slot];
  const float* p = x + arr * g.arr;
  const unsigned o = at.o[(ln.dj + 1) + 3 * (ln.dk + 1)];
  const float4 q = ld4(p, o);
  float v[6];
  v[1] = q.x; v[2] = q.y; v[3] = q.z; v[4] = q.w;
  if constexpr (quad_reads<SPT, L, -1>()) {
    v[0] = __shfl_up_sync(0xffffffffu, q.w, 1);
    if (lo) v[0] = ld_at(p, o - 4u);
  }
  if constexpr (quad_reads<SPT, L, 1>()) {
    v[5] = __shfl_down_sync(0xffffffffu, q.x, 1);
    if (hi) v[5] = ld_at(p, o + 16u);
  }
  ([&] {
    constexpr gen::TermE te = SPT::terms[SPT::lines[L].e0 + I];
#pragma unroll
    for (int s = 0; s < 4; ++s)
      acc[te.part][te.seg > 0][s] = fmaf(tab.w[te.t], v[1 + s + te.di], acc[te.part][te.seg > 0][s]);
  }(), ...);
}
template <class SPT, int NP, class Tab, int... L>
__device__ __forceinline__ void quad_lines(const Geo& g, const float* __restrict__ x, const Lines<float>& at, bool lo,
                                           bool hi, const Tab& tab, float (&acc)[NP][2][4],
                                           std::integer_sequence<int, L...>) {
  (quad_line<SPT, L>(g, x, at, lo, hi, tab, acc, std::make_integer_sequence<int, SPT::lines[L].ne>{}), ...);
}

// v at the sites of mask m
__device__ __forceinline__ void quad_store(float* base, unsigned off, int m, const float (&v)[4]) {
  if (m == 15) {
    *reinterpret_cast<float4*>(reinterpret_cast<char*>(base) + off) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (m >> s & 1) ref_at(base, off + 4u * s) = v[s];
  }
}

// grid x over the quads of the padded (i, j) plane (rows j = 0 .. ny, flat), y
// = groups of kp planes.  Every lane stays to the end (the shuffles); a lane
// past the last quad repeats it and stores nothing.
template <int VARNU, int OP, class Tab>
__device__ __forceinline__ void quad_body(const uint3 bid, const QuadA& a, const Tab& tab) {
  using SPT = gen::SP<1, VARNU, OP>;
  constexpr int NP = SPT::passes[0].np;
  const Geo& g = a.g;
  const int w = g.sx >> 2, last = (g.ny + 1) * w - 1, mine = bid.x * blockDim.x + threadIdx.x;
  const int q = min(mine, last), j = q / w, i = 4 * (q - j * w) - 1, lane = threadIdx.x & 31;
  int in = 0, face = 0;                              // sites of the lattice; those on its i faces
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (i + s >= 0 && i + s <= g.nx) in |= 1 << s;
    if (i + s == 0 || i + s == g.nx) face |= 1 << s;
  }
  if (mine > last) in = 0;
  // the lane's first (last) value has its neighbour outside the warp, and a site reads it
  const bool lo = lane == 0 && i >= 0, hi = lane == 31 && i + 3 <= g.nx;
  const bool jface = j == 0 || j == g.ny;
  const int k0 = bid.y * a.kp, k1 = min(k0 + a.kp, g.nz + 1);
  Lines<float> at(g, unsigned(i + 1) + unsigned(j + 1) * unsigned(g.sx) + unsigned(k0 + 1) * unsigned(g.sy));
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    float acc[NP][2][4] = {};
    quad_lines<SPT>(g, a.x, at, lo, hi, tab, acc, std::make_integer_sequence<int, SPT::NL>{});
    const bool jkface = jface || k == 0 || k == g.nz;
    const int bnd = (jkface ? 15 : face) & in, inner = in & ~bnd;
    const unsigned o = at.site();
    if constexpr (OP == OP_BT) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float v[4] = {acc[c][0][0], acc[c][0][1], acc[c][0][2], acc[c][0][3]};
        if (a.b) {
          const float4 b = ld4(a.b + c * g.arr, o);
          v[0] = b.x - v[0]; v[1] = b.y - v[1]; v[2] = b.z - v[2]; v[3] = b.w - v[3];
        }
        quad_store(a.y + c * g.arr, o, inner, v);
      }
    } else {                                         // the pressure row
      constexpr int P = NP - 1;
      const float es = VARNU ? float(g.eisc[k]) : 1.0f;
      if (bnd) {
        const int cjk = 3 * (j == 0 ? 0 : j == g.ny ? 2 : 1) + 9 * (k == 0 ? 0 : k == g.nz ? 2 : 1);
        const float* p = a.x + 3 * g.arr + (o >> 2);
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if (bnd >> s & 1)
            acc[P][1][s] = c_class<SPT>(
                g, p + s, a.tabs->wc + (cjk + (i + s == 0 ? 0 : i + s == g.nx ? 2 : 1)) * SPT::NCB,
                std::make_integer_sequence<int, SPT::NCB>{});
      }
      float v[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) v[s] = fmaf(es, acc[P][1][s], acc[P][0][s]);
      const float4 b = ld4(a.b + 3 * g.arr, o), p = ld4(a.x + 3 * g.arr, o);
      const double2* ml = reinterpret_cast<const double2*>(a.inv_ml + (o >> 2));
      const double2 m0 = __ldg(ml), m1 = __ldg(ml + 1);
      v[0] = p.x - float(a.s * m0.x) * (b.x - v[0]);
      v[1] = p.y - float(a.s * m0.y) * (b.y - v[1]);
      v[2] = p.z - float(a.s * m1.x) * (b.z - v[2]);
      v[3] = p.w - float(a.s * m1.y) * (b.w - v[3]);
      quad_store(a.y, o, in, v);
    }
    const unsigned step = unsigned(g.sy) * 4u;
#pragma unroll
    for (int l = 0; l < 9; ++l) at.o[l] += step;
  }
}
template <int VARNU, int OP>
__global__ void __launch_bounds__(kQuadThreads, 3) k_quad(const __grid_constant__ QuadA a,
                                                 const __grid_constant__ QuadTab<VARNU, OP> tab) {
  quad_body<VARNU, OP>(blockIdx, a, tab);
}
// batched: the table as a device copy, read through the uniform path
template <int VARNU, int OP>
struct QuadB { QuadA a; const QuadTab<VARNU, OP>* tab; };
template <int VARNU, int OP>
__global__ void __launch_bounds__(kQuadThreads, 3) kb_quad(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<QuadB<VARNU, OP>>(items, n, bid, gd);
  quad_body<VARNU, OP>(bid, it.a.a, *it.a.tab);
}

// levels with more sites than this: at 17 million sites (variable / constant
// viscosity) B^T, the pressure step and its copy take 410 / 380 us here and 476
// / 410 us with a site per thread (uzrows.cu); at 2.1 million, 70 / 64 us and
// 72 / 64 us, and four planes a block are too few blocks (82 / 75 us)
constexpr int64_t kQuadSites = 4000000;
}  // namespace
bool quad_level(const Geo& g) {
  return int64_t(g.nx + 1) * (g.ny + 1) * (g.nz + 1) > kQuadSites && g.sx % 4 == 0;
}
namespace {
bool aligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <int VARNU, int OP>
bool launch_quad(const QuadA& q, const float* w, cudaStream_t s) {
  const Geo& g = q.g;
  if (!quad_level(g) || !aligned(q.x) || !aligned(q.b) || !aligned(q.y) || !aligned(q.inv_ml)) return false;
  QuadA a = q;
  a.kp = kQuadPlanes;
  const dim3 grd(((g.ny + 1) * (g.sx / 4) + kQuadThreads - 1) / kQuadThreads, (g.nz + a.kp) / a.kp);
  using Tab = QuadTab<VARNU, OP>;
  if (g_rec) {
    g_rec->add(reinterpret_cast<const void*>(kb_quad<VARNU, OP>), grd, dim3(kQuadThreads), 0, 1,
               QuadB<VARNU, OP>{a, static_cast<const Tab*>(g_rec->table(w, sizeof(Tab)))});
    return true;
  }
  Tab tab;
  std::copy(w, w + sizeof(tab.w) / 4, tab.w);
  ++g_launches;
  void* args[] = {&a, &tab};
  cudaLaunchKernel(reinterpret_cast<const void*>(k_quad<VARNU, OP>), grd, dim3(kQuadThreads), args, 0, s);
  return true;
}

}  // namespace

bool quad_bt(int varnu, const Geo& g, const float* w, const float* x, const float* b, float* y, cudaStream_t s) {
  const QuadA a{g, x, b, y, nullptr, nullptr, 0.0, 0};
  return varnu ? launch_quad<1, OP_BT>(a, w, s) : launch_quad<0, OP_BT>(a, w, s);
}
bool quad_pressure(int varnu, const Geo& g, const float* w, const ResTabs<float>* tabs, const float* x, const float* b,
                   float* pn, const double* inv_ml, double sc, cudaStream_t s) {
  const QuadA a{g, x, b, pn, tabs, inv_ml, sc, 0};
  return varnu ? launch_quad<1, OP_BC>(a, w, s) : launch_quad<0, OP_BC>(a, w, s);
}

}  // namespace hhg
