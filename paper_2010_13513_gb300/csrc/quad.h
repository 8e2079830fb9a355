// B^T and the pressure step, P1-P1 in FP32, four aligned sites per thread (quad.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"
#include "small.h"

namespace hhg {

// whether the level is large enough, and its pitch a multiple of four
bool quad_level(const Geo& g);
constexpr int kQuadThreads = 256, kQuadPlanes = 4;

// Each launches its rows and returns true, or returns false with nothing
// launched: another level, a vector that is not 16-byte aligned.  w: the level's weights of the operator (the FastTab
// image), tabs: device table with the C stencil per boundary class.

// y = B^T p (b = null) or y = b - B^T p at the interior sites; p the pressures of x
bool quad_bt(int varnu, const Geo& g, const float* w, const float* x, const float* b, float* y, cudaStream_t s);
// pn = p - sc inv_ml (g - (B, -C) x): the pressure step of an Uzawa iteration, pn not x's pressures
bool quad_pressure(int varnu, const Geo& g, const float* w, const ResTabs<float>* tabs, const float* x, const float* b,
                   float* pn, const double* inv_ml, double sc, cudaStream_t s);

}  // namespace hhg
