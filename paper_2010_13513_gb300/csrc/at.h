// Element access by 32-bit byte offset, and pieces that the unrolled rows share.
#pragma once

#include <utility>

#include "internal.h"

namespace hhg {

// the element at byte offset `off` from `base`; with a base that is uniform
// for the launch and an unsigned 32-bit offset (a site's place in a group
// array, below 4 GB) the address needs no 64-bit arithmetic per thread
template <class T>
__device__ __forceinline__ T ld_at(const T* base, unsigned off) {
  return __ldg(reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off));
}
template <class T>
__device__ __forceinline__ T& ref_at(T* base, unsigned off) {
  return *reinterpret_cast<T*>(reinterpret_cast<char*>(base) + off);
}
template <class T>
__device__ __forceinline__ const T& ref_at(const T* base, unsigned off) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off);
}

// A row of n terms summed by m chains of consecutive terms.  Terms whose weights
// cancel on smooth fields are neighbours in the generated order and stay in one
// chain (the pressure row of P2-P1 starts -w -w -w -3w +w +w +w): dealt out in
// turn, every chain would sum values that cancel only at the end.
// The chain of term i:
constexpr int chain_of(int i, int n, int m) { return i * m / n; }
// The term evaluated in step j of chain_steps where the chains take turns (-1:
// none): for long rows in kernels of few warps (P2-P1 level 7 with variable
// viscosity, one smoothing step with its pressure row chain after chain 2.04 ms,
// in turns 1.83 ms).
constexpr int chain_term(int j, int n, int m) {
  const int q = j % m, e = (q * n + m - 1) / m + j / m;
  return e < ((q + 1) * n + m - 1) / m ? e : -1;
}
constexpr int chain_steps(int n, int m) { return (n + m - 1) / m * m; }

// the C terms of a boundary pressure row at p: the stencil wc of its class
template <class SPT, class T, int... O>
__device__ __forceinline__ T c_class(const Geo& g, const T* __restrict__ p, const T* __restrict__ wc,
                                     std::integer_sequence<int, O...>) {
  T a = T(0);
  ((a = fma(__ldg(wc + O), __ldg(p + SPT::cbo[O].di + SPT::cbo[O].dj * g.sx + SPT::cbo[O].dk * g.sy), a)), ...);
  return a;
}

// FP64 P1-P1 arrays may exceed the 4 GB (up to 715 million sites are
// accepted): its kernels count offsets from the site's plane instead
template <int DISC, class T>
constexpr bool kByPlane = DISC == 1 && sizeof(T) == 8;

// byte offsets of a site's nine neighbouring lines (dj, dk) in any group
// array: kept in registers, so that a term's load is a uniform array base, one
// of these and an immediate (di)
template <class T>
struct Lines {
  unsigned o[9];
  __device__ __forceinline__ Lines(const Geo& g, unsigned site) {
    const unsigned at = site * unsigned(sizeof(T)), sj = unsigned(g.sx) * unsigned(sizeof(T)),
                   sk = unsigned(g.sy) * unsigned(sizeof(T));
#pragma unroll
    for (int q = 0; q < 9; ++q) o[q] = at + unsigned(q % 3 - 1) * sj + unsigned(q / 3 - 1) * sk;
  }
  __device__ __forceinline__ unsigned site() const { return o[4]; }
  template <int DI, int DJ, int DK>
  __device__ __forceinline__ T ld(const T* array) const {
    return ld_at(array + DI, o[(DJ + 1) + 3 * (DK + 1)]);
  }
  // the same for an array that the kernel also writes (no read-only path)
  template <int DI, int DJ, int DK>
  __device__ __forceinline__ T get(const T* array) const {
    return ref_at(array + DI, o[(DJ + 1) + 3 * (DK + 1)]);
  }
};

}  // namespace hhg
