// Gauss-Seidel phases of the inexact Uzawa velocity step as separate launches (gs.cu).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace hhg {

constexpr int kGsTerms = 65;       // terms of a row of A at most (the diagonal first)

// the component-0 rows of A on one level (the other components' rows are the
// same on their own arrays): weights in the order of the generated structure
// (read with a variable viscosity only) and 1 / diagonal, per group
template <class T>
struct GsRows {
  T w[8][kGsTerms];
  T inv_diag[8];
};

// One phase -- group grp, colour 0..3 of the vertex group or -1 (all sites of
// an edge group) -- on the velocity components [comp, comp + ncomp); u, rhs:
// block vectors
template <class T>
void gs_phase(int disc, int varnu, const Geo& g, const GsRows<T>& rows, int grp, int colour, T* u, const T* rhs,
              int comp, int ncomp, int threads, cudaStream_t s);

// P2: the four vertex colours of a sweep (3, 2, 1, 0 if reverse): the edge
// terms of all vertex rows first (t, three group arrays of scratch), then one
// launch per colour that adds the vertex neighbours
template <class T>
void gs_vertex_phases(int varnu, const Geo& g, const GsRows<T>& rows, bool reverse, T* u, const T* rhs, T* t,
                      int threads, cudaStream_t s);

}  // namespace hhg
