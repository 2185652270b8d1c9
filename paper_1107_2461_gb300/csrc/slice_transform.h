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

// Small FP64 fields (small_f64.cu): both plane transforms in one launch when nx
// and ny are at most kSmallN, the three z steps of the TPF in one when nz is.
// Whole solves, digit products against small kernels (us): TPT 16^3 53.6 / 35.0,
// 24^3 59.6 / 39.1, 32^3 61.6 / 45.3, 40^3 69.9 / 67.6; TPF 16^3 61.6 / 30.9, 32^3
// 67.8 / 41.1, 40^3 78.0 / 67.8 (several digit planes per MMA since took 40^3 to
// 67.8 TPT and 74.0 TPF, 32^3 to 57.5 / 43.2 and 63.6 / 39.1).  The plain
// multiply-adds grow as n^4, so the line is drawn at 32.  It does not look at the
// other extents, and fields with many planes of 32 x 32 cells or z columns of 32 lie
// on the wrong side of it: TPT 16 x 16 x 256 111 / 94, 32 x 32 x 64 67.0 / 59.5, but
// 32 x 32 x 128 86 / 90, 32 x 32 x 256 135 / 152; TPF 64 x 64 x 32 73.9 / 71.9, but
// 128 x 128 x 32 127 / 144, 256 x 256 x 32 852 / 1056.
constexpr int kSmallN = 32;
bool small_plane_f64(const Field& f);
bool small_z_f64(const Field& f);
fdi_status launch_small_plane(fdi_plan* p, const Field& f, bool forward, const double* in, double* out,
                              bool accumulate, bool pdl, const int* skip, cudaStream_t s);
// forward z transform, divide and back z transform, in place
fdi_status launch_small_z(fdi_plan* p, const Field& f, double sigma, double lambda, double* data, const int* skip,
                          cudaStream_t s);

}  // namespace fdi
