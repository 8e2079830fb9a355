// Transfers between two levels (Sec. 3.3): x_f += I x_c and r_c = I^T r_f with
// the nodal (linear P1, quadratic P2) interpolation of the Kuhn lattice.
//
// The interpolation is the same in every coarse lattice cell: a fine DoF at
// doubled fine position 4 a + p (a the cell, 0 <= p_d < 4; P1: 2 a + p,
// 0 <= p_d < 2) reads the 27 (8) coarse nodes of its cell with weights that
// depend on p only.  The weights are evaluated at compile time and every
// row is unrolled over its non-zero ones, so that no table is read:
//  * prolongation: one thread owns one coarse cell and one z position p_z of
//    it, loads the coarse nodes once and updates 16 fine DoFs of a component
//    (P1 fields: all 8 of the cell), as 8 aligned pairs of sites on levels
//    with an even pitch (single sites lie two apart in the lanes);
//  * restriction: one thread gathers one coarse DoF of one group (the blocks
//    of a launch that run at the same time share the fine planes they read).
// All components, groups and the pressure go in one launch (grid z).
//
// Bound: HBM on the large levels (the fine vector is read and written, or
// read, once), launch latency on the small ones.  The table-driven kernels
// these replace read a weight and an offset per term from memory (dependent
// loads), divided a row's terms over lanes and took two launches each.
// Measured (FP32, P2-P1, 2x1x1 cubes at level 6, restriction and prolongation):
// 248 us before, 61 us now (79 us with single sites instead of pairs); their
// vectors once over HBM would take 26 us.  Level 7: restriction 372 us before,
// 92 us now; prolongation 558 us before, 127 us now.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>
#include <utility>

#include "batch.h"
#include "kernels.h"

namespace hhg {
namespace {

// local node I (the vertices, then the edges 01 02 03 12 13 23) of the Kuhn
// tetrahedron that holds the point with coordinates (px, py, pz) / 4 of a cell:
// its doubled position (0..2) in the cell and its weight at the point, quadratic
// interpolation.  The tetrahedron is 0 -> e_a -> e_a + e_b -> (1, 1, 1) of the
// coordinates in descending order.
struct P2Node { int x, y, z; double w; };
constexpr P2Node p2_node(int px, int py, int pz, int I) {
  const int p[3] = {px, py, pz};
  int o[3] = {0, 1, 2};
  for (int r = 0; r < 2; ++r)                      // stable sort, descending
    for (int s = 0; s < 2; ++s)
      if (p[o[s]] < p[o[s + 1]]) {
        const int t = o[s];
        o[s] = o[s + 1];
        o[s + 1] = t;
      }
  const double lam[4] = {(4 - p[o[0]]) / 4.0, (p[o[0]] - p[o[1]]) / 4.0, (p[o[1]] - p[o[2]]) / 4.0, p[o[2]] / 4.0};
  int v[4][3] = {};
  for (int s = 0; s < 3; ++s)
    for (int d = 0; d < 3; ++d) v[s + 1][d] = v[s][d] + (d == o[s] ? 1 : 0);
  const int a = I < 4 ? I : I < 7 ? 0 : I < 9 ? 1 : 2, b = I < 4 ? I : I < 7 ? I - 3 : I < 9 ? I - 5 : 3;
  return P2Node{v[a][0] + v[b][0], v[a][1] + v[b][1], v[a][2] + v[b][2],
                a == b ? lam[a] * (2 * lam[a] - 1) : 4 * lam[a] * lam[b]};
}
// weight of the coarse node at doubled position (nx, ny, nz) of a cell at the point
constexpr double p2_weight(int px, int py, int pz, int nx, int ny, int nz) {
  for (int I = 0; I < 10; ++I) {
    const P2Node n = p2_node(px, py, pz, I);
    if (n.x == nx && n.y == ny && n.z == nz) return n.w;
  }
  return 0.0;
}
// group of a parity offset (order of kGroupOff)
constexpr int group_at(int ox, int oy, int oz) {
  constexpr int g[8] = {0, 1, 2, 4, 3, 5, 6, 7};
  return g[ox | oy << 1 | oz << 2];
}

__device__ __forceinline__ int64_t xsite(const Geo& g, int i, int j, int k) {
  return int64_t(i + 1) + int64_t(j + 1) * g.sx + int64_t(k + 1) * g.sy;
}

// ------------------------------------------------------------- prolongation
// the value at point (PX, PY, PZ) from the loaded nodes c, NX of them in x of
// which the cell's start at X0; the small vertex terms before the edge terms
template <int PX, int PY, int PZ, int NX, int X0, int NC, class T, int... I>
__device__ __forceinline__ T p2_point(const T (&c)[NC], std::integer_sequence<int, I...>) {
  T a = T(0);
  ([&] {
    constexpr P2Node n = p2_node(PX, PY, PZ, I);
    if constexpr (n.w != 0.0) a = fma(T(n.w), c[X0 + n.x + NX * (n.y + 3 * n.z)], a);
  }(), ...);
  return a;
}
constexpr auto kP2Nodes = std::make_integer_sequence<int, 10>{};

// xf += v, or xf = v (SET)
template <bool SET, class T>
__device__ __forceinline__ void put(T* f, T v) {
  if (SET) *f = v;
  else *f += v;
}

// the 16 fine DoFs of one component at z position PZ of coarse cell (ax, ay, az)
template <int PZ, bool SET, class T, int... Q>
__device__ __forceinline__ void prolong_p2(const Geo& gf, const Geo& gc, int ax, int ay, int az, bool interior_only,
                                           const T* __restrict__ xc, T* __restrict__ xf,
                                           std::integer_sequence<int, Q...>) {
  constexpr int NZ = PZ == 0 ? 1 : 3;
  T c[NZ * 9];
  const T* x0 = xc + xsite(gc, ax, ay, az);
#pragma unroll
  for (int n = 0; n < NZ * 9; ++n) {
    const int nx = n % 3, ny = n / 3 % 3, nz = n / 9;
    c[n] = __ldg(x0 + group_at(nx & 1, ny & 1, nz & 1) * gc.arr + (nx >> 1) + (ny >> 1) * gc.sx + (nz >> 1) * gc.sy);
  }
  // doubled fine position of the point and its range: 1 .. 2 n - 1 inside
  const int lo = interior_only ? 1 : 0;
  const int Pz = 4 * az + PZ;
  if (Pz > 2 * gf.nz) return;
  const bool inz = Pz >= lo && Pz <= 2 * gf.nz - lo;
  T* f0 = xf + xsite(gf, 2 * ax, 2 * ay, 2 * az);
  auto at = [&](auto qc) {
    constexpr int q = decltype(qc)::value, PX = q % 4, PY = q / 4;
    const int Px = 4 * ax + PX, Py = 4 * ay + PY;
    if (Px > 2 * gf.nx || Py > 2 * gf.ny) return;
    const bool in = inz && Px >= lo && Px <= 2 * gf.nx - lo && Py >= lo && Py <= 2 * gf.ny - lo;
    T* f = f0 + group_at(PX & 1, PY & 1, PZ & 1) * gf.arr + (PX >> 1) + (PY >> 1) * gf.sx + (PZ >> 1) * gf.sy;
    const T v = p2_point<PX, PY, PZ, 3, 0>(c, kP2Nodes);
    if (in) put<SET>(f, v);
    else if (SET) *f = T(0);                       // Dirichlet row
  };
  (at(std::integral_constant<int, Q>{}), ...);
}

// the 8 fine DoFs of one P1 field in coarse cell (ax, ay, az)
template <bool SET, class T>
__device__ __forceinline__ void prolong_p1(const Geo& gf, const Geo& gc, int ax, int ay, int az, bool interior_only,
                                           const T* __restrict__ xc, T* __restrict__ xf) {
  T c[8];
  const T* x0 = xc + xsite(gc, ax, ay, az);
#pragma unroll
  for (int n = 0; n < 8; ++n) c[n] = __ldg(x0 + (n & 1) + (n >> 1 & 1) * gc.sx + (n >> 2) * gc.sy);
  const int lo = interior_only ? 1 : 0;
  T* f0 = xf + xsite(gf, 2 * ax, 2 * ay, 2 * az);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int px = q & 1, py = q >> 1 & 1, pz = q >> 2;
    const int i = 2 * ax + px, j = 2 * ay + py, k = 2 * az + pz;
    if (i > gf.nx || j > gf.ny || k > gf.nz) continue;
    const bool in = i >= lo && i <= gf.nx - lo && j >= lo && j <= gf.ny - lo && k >= lo && k <= gf.nz - lo;
    T* f = f0 + px + py * gf.sx + pz * gf.sy;
    if (in) put<SET>(f, q == 0 ? c[0] : T(0.5) * c[0] + T(0.5) * c[q]);
    else if (SET) *f = T(0);
  }
}

// Two fine sites of a row at a time, on levels with an even pitch: sites 2 a -
// 1 and 2 a share an aligned pair, so that a thread owns the x positions 2, 3
// of cell a - 1 and 0, 1 of cell a.  Sites outside the field's range (the halo
// column, the row padding) are rewritten as they are, or as 0 (SET).
template <class T> struct Pair2 { using type = float2; };
template <> struct Pair2<double> { using type = double2; };
template <bool SET, class T>
__device__ __forceinline__ void put_pair(T* f, bool in0, bool in1, T v0, T v1) {
  using P = typename Pair2<T>::type;
  P p;
  if (!SET) p = *reinterpret_cast<const P*>(f);
  else p.x = p.y = T(0);
  if (in0) p.x += v0;
  if (in1) p.y += v1;
  *reinterpret_cast<P*>(f) = p;
}
template <int PZ, bool SET, class T, int... Q>
__device__ __forceinline__ void prolong_p2_pair(const Geo& gf, const Geo& gc, int ax, int ay, int az,
                                                bool interior_only, const T* __restrict__ xc, T* __restrict__ xf,
                                                std::integer_sequence<int, Q...>) {
  constexpr int NZ = PZ == 0 ? 1 : 3;
  T c[NZ * 15];
  const T* x0 = xc + xsite(gc, ax - 1, ay, az);
#pragma unroll
  for (int n = 0; n < NZ * 15; ++n) {
    const int nx = n % 5, ny = n / 5 % 3, nz = n / 15;
    c[n] = __ldg(x0 + group_at(nx & 1, ny & 1, nz & 1) * gc.arr + (nx >> 1) + (ny >> 1) * gc.sx + (nz >> 1) * gc.sy);
  }
  const int lo = interior_only ? 1 : 0;
  const int Pz = 4 * az + PZ;
  if (Pz > 2 * gf.nz) return;
  const bool inz = Pz >= lo && Pz <= 2 * gf.nz - lo;
  T* f0 = xf + xsite(gf, 2 * ax - 1, 2 * ay, 2 * az);
  auto at = [&](auto qc) {
    constexpr int q = decltype(qc)::value, ODD = q & 1, PY = q >> 1;
    const int Px = 4 * ax + ODD, Py = 4 * ay + PY;
    if (Py > 2 * gf.ny) return;
    const bool in = inz && Py >= lo && Py <= 2 * gf.ny - lo;
    if (!SET && !in) return;
    T* f = f0 + group_at(ODD, PY & 1, PZ & 1) * gf.arr + (PY >> 1) * gf.sx + (PZ >> 1) * gf.sy;
    put_pair<SET>(f, in && Px - 2 >= lo && Px - 2 <= 2 * gf.nx - lo, in && Px >= lo && Px <= 2 * gf.nx - lo,
                  p2_point<2 + ODD, PY, PZ, 5, 0>(c, kP2Nodes), p2_point<ODD, PY, PZ, 5, 2>(c, kP2Nodes));
  };
  (at(std::integral_constant<int, Q>{}), ...);
}
template <bool SET, class T>
__device__ __forceinline__ void prolong_p1_pair(const Geo& gf, const Geo& gc, int ax, int ay, int az,
                                                bool interior_only, const T* __restrict__ xc, T* __restrict__ xf) {
  T c[8];                                          // x nodes a - 1 and a
  const T* x0 = xc + xsite(gc, ax - 1, ay, az);
#pragma unroll
  for (int n = 0; n < 8; ++n) c[n] = __ldg(x0 + (n & 1) + (n >> 1 & 1) * gc.sx + (n >> 2) * gc.sy);
  const int lo = interior_only ? 1 : 0;
  T* f0 = xf + xsite(gf, 2 * ax - 1, 2 * ay, 2 * az);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int py = q & 1, pz = q >> 1, i = 2 * ax, j = 2 * ay + py, k = 2 * az + pz;
    if (j > gf.ny || k > gf.nz) continue;
    const bool in = j >= lo && j <= gf.ny - lo && k >= lo && k <= gf.nz - lo;
    if (!SET && !in) continue;
    put_pair<SET>(f0 + py * gf.sx + pz * gf.sy, in && i - 1 >= lo && i - 1 <= gf.nx - lo,
                  in && i >= lo && i <= gf.nx - lo, T(0.5) * c[0] + T(0.5) * c[1 + 2 * q],
                  q == 0 ? c[1] : T(0.5) * c[1] + T(0.5) * c[1 + 2 * q]);
  }
}

// arguments of both transfers (in: coarse and out: fine for the prolongation,
// the other way round for the restriction); interior_only: Dirichlet velocity
// DoFs are left as they are
template <class T>
struct TransferA { Geo gf, gc; int interior_only; const T* in; T* out; };

// grid: x over the (i, j) plane of coarse cells (flat), z = plane and part
// (part fastest: blocks that run together share the coarse planes)
template <int PZ, bool SET, bool PAIR, class T>
__device__ __forceinline__ void prolong_p2_z(const Geo& gf, const Geo& gc, int ax, int ay, int az, bool io,
                                             const T* xc, T* xf) {
  if constexpr (PAIR) prolong_p2_pair<PZ, SET>(gf, gc, ax, ay, az, io, xc, xf, std::make_integer_sequence<int, 8>{});
  else prolong_p2<PZ, SET>(gf, gc, ax, ay, az, io, xc, xf, std::make_integer_sequence<int, 16>{});
}
template <bool SET, bool PAIR, class T>
__device__ __forceinline__ void prolong_field(const Geo& gf, const Geo& gc, int ax, int ay, int az, bool io,
                                              const T* xc, T* xf) {
  if constexpr (PAIR) prolong_p1_pair<SET>(gf, gc, ax, ay, az, io, xc, xf);
  else prolong_p1<SET>(gf, gc, ax, ay, az, io, xc, xf);
}
template <int G, bool SET, bool PAIR, class T>
__device__ __forceinline__ void prolong_body(const uint3 bid, const TransferA<T>& a) {
  constexpr int NPART = G == 8 ? 13 : 4;
  const Geo &gf = a.gf, &gc = a.gc;
  const int az = int(bid.z) / NPART, part = int(bid.z) - az * NPART;
  const int w = gc.nx + 1, q = bid.x * blockDim.x + threadIdx.x;
  const int ay = q / w, ax = q - ay * w;
  if (ay > gc.ny) return;
  const bool io = a.interior_only != 0;
  if constexpr (G == 1) {
    prolong_field<SET, PAIR>(gf, gc, ax, ay, az, io && part < 3, a.in + part * gc.arr, a.out + part * gf.arr);
  } else {
    if (part == 12) return prolong_field<SET, PAIR>(gf, gc, ax, ay, az, false, a.in + 24 * gc.arr, a.out + 24 * gf.arr);
    const int comp = part >> 2;
    const T* xc = a.in + comp * 8 * gc.arr;
    T* xf = a.out + comp * 8 * gf.arr;
    switch (part & 3) {
      case 0: prolong_p2_z<0, SET, PAIR>(gf, gc, ax, ay, az, io, xc, xf); break;
      case 1: prolong_p2_z<1, SET, PAIR>(gf, gc, ax, ay, az, io, xc, xf); break;
      case 2: prolong_p2_z<2, SET, PAIR>(gf, gc, ax, ay, az, io, xc, xf); break;
      default: prolong_p2_z<3, SET, PAIR>(gf, gc, ax, ay, az, io, xc, xf); break;
    }
  }
}

// --------------------------------------------------------------- restriction
// weight with which the coarse node of parity offset O reads the fine node at
// doubled fine distance e from it (|e| <= 3): the fine node lies in the cell
// b = floor((2 o + e) / 4) at position p = (2 o + e) mod 4
constexpr int cell_of(int t) { return t < 0 ? -1 : t / 4; }
constexpr double p2_restrict_weight(int ox, int oy, int oz, int ex, int ey, int ez) {
  const int bx = cell_of(2 * ox + ex), by = cell_of(2 * oy + ey), bz = cell_of(2 * oz + ez);
  return p2_weight(2 * ox + ex - 4 * bx, 2 * oy + ey - 4 * by, 2 * oz + ez - 4 * bz, ox - 2 * bx, oy - 2 * by,
                   oz - 2 * bz);
}

// the fine nodes around coarse node (2 a + o) with a weight: group and site
// relative to the fine vertex at the node's cell (doubled fine position 4 a), by
// group and offset (x slowest)
struct RTerm { int grp, dx, dy, dz; double w; };
struct RTerms { int n; RTerm t[125]; };
template <int OX, int OY, int OZ>
constexpr RTerms p2_restrict_terms() {
  RTerms r{};
  for (int g = 0; g < 8; ++g)
    for (int dx = -2; dx <= 2; ++dx)
      for (int dy = -2; dy <= 2; ++dy)
        for (int dz = -2; dz <= 2; ++dz) {
          const int ex = 2 * dx + kGroupOff[g][0] - 2 * OX, ey = 2 * dy + kGroupOff[g][1] - 2 * OY,
                    ez = 2 * dz + kGroupOff[g][2] - 2 * OZ;
          if (ex < -3 || ex > 3 || ey < -3 || ey > 3 || ez < -3 || ez > 3) continue;
          const double w = p2_restrict_weight(OX, OY, OZ, ex, ey, ez);
          if (w != 0.0) r.t[r.n++] = RTerm{g, dx, dy, dz, w};
        }
  return r;
}
template <int OX, int OY, int OZ>
struct Restrict { static constexpr RTerms r = p2_restrict_terms<OX, OY, OZ>(); };

// sum over the fine nodes around coarse node (2 a + o); f0: the fine vertex at
// the node's cell.  Eight chains of equal length: short sums (with chains that
// differ by the zero weights left out the FP32 error is a tenth larger) and
// independent latencies.
template <int OX, int OY, int OZ, class T, int... E>
__device__ __forceinline__ T restrict_p2(const Geo& gf, const T* __restrict__ f0, std::integer_sequence<int, E...>) {
  T s[8] = {};
  ([&] {
    constexpr RTerm t = Restrict<OX, OY, OZ>::r.t[E];
    s[E & 7] = fma(T(t.w), __ldg(f0 + t.grp * gf.arr + t.dx + t.dy * gf.sx + t.dz * gf.sy), s[E & 7]);
  }(), ...);
  return ((s[0] + s[4]) + (s[2] + s[6])) + ((s[1] + s[5]) + (s[3] + s[7]));
}

// a P1 field: two chains over the 15 fine nodes in the order of their offsets
template <class T>
__device__ __forceinline__ T restrict_p1(const Geo& gf, const T* __restrict__ f) {
  T s[2] = {T(0), T(0)};
#pragma unroll
  for (int q = 0; q < 15; ++q) {
    // 7 - q: the offsets (x, y, z) in binary below the node, its own, and above it
    const int b = q < 7 ? 7 - q : q - 7;
    const int d = (b >> 2 & 1) + (b >> 1 & 1) * gf.sx + (b & 1) * int(gf.sy);
    s[q & 1] = fma(q == 7 ? T(1) : T(0.5), __ldg(q < 7 ? f - d : f + d), s[q & 1]);
  }
  return s[0] + s[1];
}

template <int GRP, class T>
__device__ __forceinline__ void restrict_group(const Geo& gf, const Geo& gc, int i, int j, int k, const T* rf, T* rc) {
  constexpr int ox = kGroupOff[GRP][0], oy = kGroupOff[GRP][1], oz = kGroupOff[GRP][2];
  if (i > gc.nx - ox || j > gc.ny - oy || k > gc.nz - oz) return;
  const int Px = 2 * i + ox, Py = 2 * j + oy, Pz = 2 * k + oz;
  const bool inside = Px > 0 && Py > 0 && Pz > 0 && Px < 2 * gc.nx && Py < 2 * gc.ny && Pz < 2 * gc.nz;
  T v = T(0);
  if (inside)
    v = restrict_p2<ox, oy, oz>(gf, rf + xsite(gf, 2 * i, 2 * j, 2 * k),
                                std::make_integer_sequence<int, Restrict<ox, oy, oz>::r.n>{});
  rc[GRP * gc.arr + xsite(gc, i, j, k)] = v;
}

// grid: as the prolongation's, over the coarse sites; a part is one group of
// one component, or the pressure
template <int G, class T>
__device__ __forceinline__ void restrict_body(const uint3 bid, const TransferA<T>& a) {
  constexpr int NPART = 3 * G + 1;
  const Geo &gf = a.gf, &gc = a.gc;
  const int k = int(bid.z) / NPART, part = int(bid.z) - k * NPART;
  const int w = gc.nx + 1, q = bid.x * blockDim.x + threadIdx.x;
  const int j = q / w, i = q - j * w;
  if (j > gc.ny) return;
  if (G == 1 || part == 3 * G) {
    const bool zero = part < 3 * G && (i == 0 || j == 0 || k == 0 || i == gc.nx || j == gc.ny || k == gc.nz);
    T v = T(0);
    if (!zero) v = restrict_p1<T>(gf, a.in + part * gf.arr + xsite(gf, 2 * i, 2 * j, 2 * k));
    a.out[part * gc.arr + xsite(gc, i, j, k)] = v;
  } else {
    const int comp = part >> 3;
    const T* rf = a.in + comp * 8 * gf.arr;
    T* rc = a.out + comp * 8 * gc.arr;
    switch (part & 7) {
      case 0: restrict_group<0>(gf, gc, i, j, k, rf, rc); break;
      case 1: restrict_group<1>(gf, gc, i, j, k, rf, rc); break;
      case 2: restrict_group<2>(gf, gc, i, j, k, rf, rc); break;
      case 3: restrict_group<3>(gf, gc, i, j, k, rf, rc); break;
      case 4: restrict_group<4>(gf, gc, i, j, k, rf, rc); break;
      case 5: restrict_group<5>(gf, gc, i, j, k, rf, rc); break;
      case 6: restrict_group<6>(gf, gc, i, j, k, rf, rc); break;
      default: restrict_group<7>(gf, gc, i, j, k, rf, rc); break;
    }
  }
}

template <int G, bool SET, bool PAIR, class T>
__global__ void __launch_bounds__(128) k_prolong(const __grid_constant__ TransferA<T> a) {
  prolong_body<G, SET, PAIR, T>(blockIdx, a);
}
template <int G, class T>
__global__ void __launch_bounds__(128) k_restrict(const __grid_constant__ TransferA<T> a) {
  restrict_body<G, T>(blockIdx, a);
}
template <int G, bool SET, bool PAIR, class T>
__global__ void __launch_bounds__(128) kb_prolong(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<TransferA<T>>(items, n, bid, gd);
  prolong_body<G, SET, PAIR, T>(bid, it.a);
}
template <int G, class T>
__global__ void __launch_bounds__(128) kb_restrict(const void* items, int n) {
  uint3 bid, gd;
  const auto& it = batch_item<TransferA<T>>(items, n, bid, gd);
  restrict_body<G, T>(bid, it.a);
}

template <class T>
void launch(const void* kernel, const void* batched, dim3 grd, const TransferA<T>& a, cudaStream_t s) {
  const dim3 blk(128, 1, 1);
  if (g_rec) return g_rec->add(batched, grd, blk, 0, 1, a);
  ++g_launches;
  void* args[] = {const_cast<TransferA<T>*>(&a)};
  cudaLaunchKernel(kernel, grd, blk, args, 0, s);
}
inline unsigned plane_blocks(const Geo& gc) { return unsigned(((gc.nx + 1) * (gc.ny + 1) + 127) / 128); }

template <int G, bool SET, bool PAIR, class T>
void launch_prolong_as(const TransferA<T>& a, cudaStream_t s) {
  launch<T>(reinterpret_cast<const void*>(k_prolong<G, SET, PAIR, T>),
            reinterpret_cast<const void*>(kb_prolong<G, SET, PAIR, T>),
            dim3(plane_blocks(a.gc), 1, (a.gc.nz + 1) * (G == 8 ? 13 : 4)), a, s);
}
template <int G, class T>
void launch_prolong_g(const TransferA<T>& a, bool set, bool pair, cudaStream_t s) {
  if (set) pair ? launch_prolong_as<G, true, true>(a, s) : launch_prolong_as<G, true, false>(a, s);
  else pair ? launch_prolong_as<G, false, true>(a, s) : launch_prolong_as<G, false, false>(a, s);
}

}  // namespace

template <class T>
void launch_prolong(const Geo& gf, const Geo& gc, bool interior_only, bool set, const T* xc, T* xf, cudaStream_t s) {
  const TransferA<T> a{gf, gc, interior_only ? 1 : 0, xc, xf};
  // pairs of sites where they are aligned: an even pitch (levels with nx >=
  // 64 have a multiple of four, the smaller ones nx + 3) and vector
  const bool pair = gf.sx % 2 == 0 && gf.sy % 2 == 0 && reinterpret_cast<uintptr_t>(xf) % (2 * sizeof(T)) == 0;
  if (gf.G == 1) launch_prolong_g<1, T>(a, set, pair, s);
  else launch_prolong_g<8, T>(a, set, pair, s);
}

template <class T>
void launch_restrict(const Geo& gf, const Geo& gc, const T* rf, T* rc, cudaStream_t s) {
  const TransferA<T> a{gf, gc, 1, rf, rc};
  if (gf.G == 1)
    launch<T>(reinterpret_cast<const void*>(k_restrict<1, T>), reinterpret_cast<const void*>(kb_restrict<1, T>),
              dim3(plane_blocks(gc), 1, (gc.nz + 1) * 4), a, s);
  else
    launch<T>(reinterpret_cast<const void*>(k_restrict<8, T>), reinterpret_cast<const void*>(kb_restrict<8, T>),
              dim3(plane_blocks(gc), 1, (gc.nz + 1) * 25), a, s);
}

#define HHG_INST(T)                                                                               \
  template void launch_prolong<T>(const Geo&, const Geo&, bool, bool, const T*, T*, cudaStream_t); \
  template void launch_restrict<T>(const Geo&, const Geo&, const T*, T*, cudaStream_t);
HHG_INST(double)
HHG_INST(float)

}  // namespace hhg
