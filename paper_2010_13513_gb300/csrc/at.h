// Element access by 32-bit byte offset.
#pragma once

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
