// All rows of the P2-P1 operator on large levels, marching along k (march.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"

namespace hhg {

// y = calA x (MODE_SET) or y = b - calA x (MODE_RES) over all rows of a level
// (Dirichlet velocity rows 0); inputs with zero Dirichlet velocity entries.
// tab: host FastTab of the full operator (read with a variable viscosity
// only)
template <class T>
void march_rows(int varnu, int mode, const Geo& g, const void* tab, const T* x, const T* b, T* y, cudaStream_t s);

}  // namespace hhg
