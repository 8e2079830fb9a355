// Tables and launch shapes of the specialised stencil kernels (rows.cu,
// march.cu, stream.cu, gs.cu): their row structure is known at compile time.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace hhg {

// weights and linear offsets (array * array_stride + di + dj sx + dk sy) of
// the interior terms of one operator on one level, in table order
template <class T, int N>
struct FastTab {
  T w[N];
  int off[N];
};

// launch shape of the specialised kernels on one level (autotuned)
struct Shape {
  int row_threads = 128;   // reported by hhg_get_launch_shape; the row kernels have one shape
  int row_kplanes = 2;
  int row_sites = 1;
  int gs_threads = 128;    // threads per block of the Gauss-Seidel kernels
  int gs_lanes = 1;        // reported by hhg_get_launch_shape; a Gauss-Seidel site has one lane
  int gs_threads0 = 0;     // threads per block of the vertex colour phases (0 = gs_threads)
  // streaming kernels (stream.cu) of the full operator: threads per block (0 =
  // the unstaged rows), in the V-cycle precision (st_threads) and in FP64
  // (st64_threads; the mixed solve's outer residual)
  int st_threads = 0;
  int st64_threads = 0;
  int st_sites = 4;        // sites per thread of the FP32 streaming kernels (2 or 4)
  // order of the per-phase Gauss-Seidel launches of a smoothing step: 0 = every
  // phase on the three components at once; 1 = component by component (all
  // sweeps of one component before the next: its arrays stay in L2 on levels
  // whose vectors exceed it)
  int gs_comp_major = 0;
  int gs_edge_sums = 0;    // P2: the vertex colours on shared edge sums (gs_vertex_phases)
};

// number of interior terms of a specialised operator (-1 if none)
int fast_terms(int disc, int varnu, int op);

}  // namespace hhg
