// Weights of the constant-viscosity rows, and the power of h they are scaled by.
//
// At h = 1 the weights of A are multiples of 1 / 15 (P2-P1) or 1 (P1-P1), those
// of B and B^T of 1 / 60 or 1 / 12, those of C of one irrational unit (it has
// |T|^(2/3)).  FP32 rows take them as small integers, which are exact, and the
// factor (h / K, h^2 / K, h^3 times the unit, 1 / diagonal) once per row in two
// parts: rounded to FP32 it would be a relative error of up to 6e-8 common to
// all rows, which the sweeps of a smoother add up (P2-P1 level 5, a smoothing
// step: velocity error 1.0e-7 with weights rounded one by one, 1.9e-7 with
// integers and a rounded 1 / diagonal, 7.4e-8 now).  FP64 rows take the weights of h = 1 and
// a rounded factor.
#pragma once

#include <cstdint>

namespace hhg {

template <int DISC> constexpr double kScaleA = DISC == 2 ? 15.0 : 1.0;
template <int DISC> constexpr double kScaleB = DISC == 2 ? 60.0 : 12.0;
constexpr double rounded(double v) { return v < 0 ? -double(int64_t(0.5 - v)) : double(int64_t(v + 0.5)); }
constexpr bool near_integer(double v) {
  const double d = v - rounded(v);
  return d < 1e-9 && d > -1e-9;
}
// term E of operator table S as a row of T holds it, and what its factor is
// divided by; K: the scale that makes it an integer
template <class S, int E, class T>
constexpr double row_weight(double K) {
  return sizeof(T) == 4 ? rounded(S::wref[E] * K) : S::wref[E];
}
template <class T>
constexpr double row_scale(double K) { return sizeof(T) == 4 ? K : 1.0; }

// a factor > 0.  FP32: the low part is always positive (the high one is a little
// too small), so that an infinite sum stays one
template <class T>
struct Factor { T hi, lo; };
template <class T>
constexpr Factor<T> make_factor(double v) {
  if (sizeof(T) == 8) return {T(v), T(0)};
  const T hi = T(v * (1.0 - 1.0 / (1 << 22)));
  return {hi, T(v - double(hi))};
}
// f s and r - f s, the low part first: what is left is rounded once, and a
// constant stays one in a Gauss-Seidel row (an error that all updates of a smooth
// vector share would add up over the sweeps)
template <class T>
__device__ __forceinline__ T scaled(const Factor<T>& f, T s) {
  if constexpr (sizeof(T) == 8) return f.hi * s;
  else return fma(f.hi, s, f.lo * s);
}
template <class T>
__device__ __forceinline__ T minus_scaled(T r, const Factor<T>& f, T s) {
  if constexpr (sizeof(T) == 8) return fma(-f.hi, s, r);
  else return fma(-f.hi, s, fma(-f.lo, s, r));
}

// whether the weights E0 .. E0 + n - 1 times K are small integers
template <class S>
constexpr bool int_weights(int E0, int n, double K) {
  for (int e = E0; e < E0 + n; ++e)
    if (!near_integer(S::wref[e] * K) || S::wref[e] * K > 1024.0 || S::wref[e] * K < -1024.0) return false;
  return true;
}
// the unit of the C terms E0 .. E0 + n - 1 at h = 1: a sixth of the diagonal's weight
template <class S>
constexpr double c_unit(int E0, int n) {
  for (int e = E0; e < E0 + n; ++e)
    if (S::off[e].di == 0 && S::off[e].dj == 0 && S::off[e].dk == 0) return (S::wref[e] < 0 ? -S::wref[e] : S::wref[e]) / 6.0;
  return 1.0;
}

}  // namespace hhg
