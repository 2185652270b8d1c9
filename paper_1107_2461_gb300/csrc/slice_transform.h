// FP64 eigenvector transforms on the tensor cores by exact digit products:
// declarations shared by the plan and the solver.
#pragma once
#include <cuda_runtime.h>

#include "fdi_internal.h"

namespace fdi {

// A transform matrix T (n x n, output index k, input index j) as base-256
// digits: eight fp16 digit planes of every row, already in the layout the
// MMA reads ([128-row tile][16-column chunk][digit][row][column], 32-byte
// swizzle), and the biased exponent of each row's largest entry.
struct SliceMatrix {
  int n = 0, m_tiles = 0, n_chunks = 0;
  unsigned char* img = nullptr;
  int* row_exp = nullptr;
};

struct SliceAxis {
  SliceMatrix fwd, bwd;  // E^{-1}, E
};

// Geometry of the lines a transform contracts: line r < R starts at
// (r / S) * slab + (r % S) * rs, element j of it at + j * ks (input and output).
struct SliceLines {
  long long R = 0, S = 1, slab = 0, rs = 0, ks = 0;
};

fdi_status slice_prepare_axis(fdi_plan* p, Axis* ax, cudaStream_t s);
void slice_free_axis(Axis* ax);
// out (+)= T in along every line; in and out distinct
fdi_status launch_slice_transform(fdi_plan* p, const SliceMatrix& m, const double* in, double* out,
                                  const SliceLines& g, bool accumulate, bool pdl, const int* skip,
                                  cudaStream_t s);

}  // namespace fdi
