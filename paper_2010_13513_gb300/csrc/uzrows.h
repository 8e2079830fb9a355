// Row evaluations of an Uzawa iteration that runs as separate launches (uzrows.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"
#include "small.h"

namespace hhg {

// y_u = B^T p (MODE_SET) or b_u - B^T p (MODE_RES) at the interior velocity
// rows (Dirichlet rows of y are left as they are); w: the weights of B^T in
// the order of the generated structure (read with a variable viscosity only)
template <class T>
void bt_rows(int disc, int varnu, int mode, const Geo& g, const T* w, const T* x, const T* b, T* y, cudaStream_t s);

// p -= s M_L^{-1} (g - (B u - C p)) at every pressure site of x, g = b_p; w:
// the weights of (B, -C); tabs: device table with the C stencil per boundary
// class; tmp: scratch block vector (P1-P1: its pressure array is overwritten)
template <class T>
void uzawa_pressure(int disc, int varnu, const Geo& g, const T* w, const ResTabs<T>* tabs, T* x, const T* b, T* tmp,
                    const double* inv_mlhat, double s, cudaStream_t st);

// launch shapes of the two on a level (fp32: the precision), for reports
struct RowsShape { int threads, planes, sites; };
RowsShape bt_shape(int disc, bool fp32, const Geo& g);
RowsShape pressure_shape(int disc, bool fp32, const Geo& g);

// y_p = B u - C p, FP64 (the power iteration of the spectral estimate); w, tabs
// as above
void bc_rows(int disc, int varnu, const Geo& g, const double* w, const ResTabs<double>* tabs, const double* x,
             double* y, cudaStream_t s);

}  // namespace hhg
