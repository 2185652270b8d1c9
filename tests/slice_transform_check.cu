// One FP64 digit transform of libfdi.so on caller-supplied device arrays, for
// test_gpu_slice_exact.py: prepares the digit planes of T (n x n) and applies it
// to `lines` lines of in (out (+)= T in along every line).  contiguous: line r is
// in[r * n ..]; else the lines of [slab][n][width] with `width` neighbouring lines.
#include "fdi_internal.h"
#include "slice_transform.h"

// status of preparing an n x n matrix, n so large that its digit planes exceed any
// device memory: the allocation is refused before anything reads T
extern "C" int slice_prepare_status(int n) {
  fdi_plan p;
  fdi::Axis ax;
  ax.n = n;
  const int st = (int)fdi::slice_prepare_axis(&p, &ax, nullptr);
  fdi::slice_free_axis(&ax);
  return st;
}

extern "C" int slice_transform_check(const double* T, int n, const double* in, double* out, long long lines,
                                     int contiguous, long long width, int accumulate) {
  fdi_plan p;
  if (cudaGetDevice(&p.device) != cudaSuccess) return -1;
  if (cudaMalloc(&p.d_err, sizeof(int)) != cudaSuccess) return -2;
  int err = -3;
  fdi::Axis ax;
  ax.n = n;
  ax.E = ax.Einv = const_cast<double*>(T);
  fdi::SliceLines g;
  g.R = lines;
  g.S = contiguous ? lines : width;
  g.slab = contiguous ? 0 : width * n;
  g.rs = contiguous ? n : 1;
  g.ks = contiguous ? 1 : width;
  if (cudaMemset(p.d_err, 0, sizeof(int)) == cudaSuccess && fdi::slice_prepare_axis(&p, &ax, nullptr) == FDI_OK &&
      fdi::launch_slice_transform(&p, static_cast<fdi::SliceAxis*>(ax.slices)->fwd, in, out, g, accumulate != 0, false,
                                  nullptr, nullptr) == FDI_OK &&
      cudaDeviceSynchronize() == cudaSuccess)
    cudaMemcpy(&err, p.d_err, sizeof(int), cudaMemcpyDeviceToHost);
  fdi::slice_free_axis(&ax);
  cudaFree(p.d_err);
  return err;
}
