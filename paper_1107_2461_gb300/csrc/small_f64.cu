// FP64 transforms of small fields: both plane transforms of a z-plane, or the z
// transforms and the spectral divide of a group of columns, in one launch.
//
// On a field with few cells per direction a transform launch is all latency (a
// 16^3 pass through the digit products takes 6 us for 0.1 us of work), and plain
// FP64 multiply-adds (2 lanes per clock and SM) are fast enough: the work of one
// plane is split over as many CTAs as it takes, without recomputing anything.
//   forward (Eq. 25 along x, then y): a CTA takes kSmallCols of the nx x-modes of
//     a plane: F1[y][i] = sum_x Ex^-1[i][x] f[y][x], F2[j][i] = sum_y Ey^-1[j][y] F1[y][i]
//   back (y, then x): a CTA takes kSmallCols of the ny rows:
//     G[y][i] = sum_j Ey[y][j] F[j][i], u[y][x] = sum_i Ex[x][i] G[y][i]
//   z (TPF, Eq. 26-29): a CTA takes kSmallCols (y, x) columns: forward, divide by
//     sigma - lambda (Lx + Ly + Lz), back
// Matrices and data sit in shared memory; the matrices (plan data) are loaded
// before the wait for the previous kernel.
#include "fdi_internal.h"
#include "slice_transform.h"

namespace fdi {
namespace {

constexpr int kSmallCols = 4;
constexpr int kSmallThreads = 128;

struct SmallArgs {
  const double* in;
  double* out;
  const double* Tx;  // nx x nx
  const double* Ty;  // ny x ny
  int nx, ny;
  int accumulate;
};

// C[r][c] = sum_k A[r * as + k] B[k * bs + c] for r < nr, c < nc, by the block's threads
template <typename Store>
__device__ __forceinline__ void small_product(const double* A, int as, int nr, const double* B, int bs, int nc, int K,
                                              Store&& store) {
  for (int e = threadIdx.x; e < nr * nc; e += kSmallThreads) {
    const int r = e / nc, c = e - r * nc;
    const double* a = A + r * as;
    const double* b = B + c;
    double s = 0.0;
#pragma unroll 4
    for (int k = 0; k < K; ++k) s = fma(a[k], b[k * bs], s);
    store(r, c, s);
  }
}

// rows padded to an odd number of doubles: columns of a tile spread over the banks
__host__ __device__ constexpr int odd(int n) { return n | 1; }

// blockIdx.x: group of x-modes, blockIdx.y: plane
__global__ void __launch_bounds__(kSmallThreads) k_small_forward(const SmallArgs a, const int* __restrict__ skip) {
  extern __shared__ double sm[];
  const int nx = a.nx, ny = a.ny, px = odd(nx), py = odd(ny);
  const int i0 = blockIdx.x * kSmallCols, nc = min(kSmallCols, nx - i0);
  double* sTx = sm;                        // [x][nc]: rows i0.. of Ex^-1, transposed
  double* sTy = sTx + nx * kSmallCols;     // [j][py]
  double* sf = sTy + ny * py;              // [y][px]
  double* s1 = sf + ny * px;               // [y][nc]
  for (int e = threadIdx.x; e < nc * nx; e += kSmallThreads) {
    const int i = e / nx, x = e - i * nx;
    sTx[x * kSmallCols + i] = a.Tx[(i0 + i) * nx + x];
  }
  for (int e = threadIdx.x; e < ny * ny; e += kSmallThreads) sTy[(e / ny) * py + e % ny] = a.Ty[e];
  pdl_wait();
  if (skip && *skip) return;
  const long long base = (long long)blockIdx.y * ny * nx;
  for (int e = threadIdx.x; e < ny * nx; e += kSmallThreads) sf[(e / nx) * px + e % nx] = a.in[base + e];
  __syncthreads();
  small_product(sf, px, ny, sTx, kSmallCols, nc, nx, [&](int y, int i, double v) { s1[y * kSmallCols + i] = v; });
  __syncthreads();
  small_product(sTy, py, ny, s1, kSmallCols, nc, ny,
                [&](int j, int i, double v) { a.out[base + (long long)j * nx + i0 + i] = v; });
}

// blockIdx.x: group of rows y, blockIdx.y: plane
__global__ void __launch_bounds__(kSmallThreads) k_small_back(const SmallArgs a, const int* __restrict__ skip) {
  extern __shared__ double sm[];
  const int nx = a.nx, ny = a.ny, px = odd(nx);
  const int y0 = blockIdx.x * kSmallCols, nr = min(kSmallCols, ny - y0);
  double* sTx = sm;                   // [i][px]: Ex transposed
  double* sTy = sTx + nx * px;        // [nr][ny]
  double* sF = sTy + kSmallCols * ny; // [j][px]
  double* s1 = sF + ny * px;          // [nr][px]
  for (int e = threadIdx.x; e < nx * nx; e += kSmallThreads) sTx[(e % nx) * px + e / nx] = a.Tx[e];
  for (int e = threadIdx.x; e < nr * ny; e += kSmallThreads) sTy[e] = a.Ty[y0 * ny + e];
  pdl_wait();
  if (skip && *skip) return;
  const long long base = (long long)blockIdx.y * ny * nx;
  for (int e = threadIdx.x; e < ny * nx; e += kSmallThreads) sF[(e / nx) * px + e % nx] = a.in[base + e];
  __syncthreads();
  small_product(sTy, ny, nr, sF, px, nx, ny, [&](int y, int i, double v) { s1[y * px + i] = v; });
  __syncthreads();
  small_product(s1, px, nr, sTx, px, nx, nx, [&](int y, int x, double v) {
    double* dst = a.out + base + (long long)(y0 + y) * nx + x;
    *dst = a.accumulate ? *dst + v : v;
  });
}

struct SmallZArgs {
  double* data;  // in place
  const double* Tf;
  const double* Tb;
  const double* lx;
  const double* ly;
  const double* lz;
  int nx, ny, nz, singular;
  double sigma, lambda;
};

__global__ void __launch_bounds__(kSmallThreads) k_small_z(const SmallZArgs a, const int* __restrict__ skip) {
  extern __shared__ double sm[];
  const int nz = a.nz, pz = odd(nz), plane = a.nx * a.ny;
  const int c0 = blockIdx.x * kSmallCols, nc = min(kSmallCols, plane - c0);
  double* sTf = sm;                 // [k][pz]
  double* sTb = sTf + nz * pz;      // [k][pz]
  double* sf = sTb + nz * pz;       // [z][kSmallCols]
  double* s1 = sf + nz * kSmallCols;
  for (int e = threadIdx.x; e < nz * nz; e += kSmallThreads) {
    sTf[(e / nz) * pz + e % nz] = a.Tf[e];
    sTb[(e / nz) * pz + e % nz] = a.Tb[e];
  }
  pdl_wait();
  if (skip && *skip) return;
  for (int e = threadIdx.x; e < nz * nc; e += kSmallThreads) {
    const int z = e / nc, c = e - z * nc;
    sf[z * kSmallCols + c] = a.data[(long long)z * plane + c0 + c];
  }
  __syncthreads();
  small_product(sTf, pz, nz, sf, kSmallCols, nc, nz, [&](int k, int c, double v) {
    const int col = c0 + c;
    const double ls = a.lx[col % a.nx] + a.ly[col / a.nx] + a.lz[k];
    s1[k * kSmallCols + c] = (a.singular && ls == 0.0) ? 0.0 : v / (a.sigma - a.lambda * ls);
  });
  __syncthreads();
  small_product(sTb, pz, nz, s1, kSmallCols, nc, nz,
                [&](int z, int c, double v) { a.data[(long long)z * plane + c0 + c] = v; });
}

size_t plane_bytes(int nx, int ny) {
  // the larger of the two kernels' layouts
  const size_t fwd = (size_t)nx * kSmallCols + (size_t)ny * odd(ny) + (size_t)ny * odd(nx) + (size_t)ny * kSmallCols;
  const size_t back = (size_t)nx * odd(nx) + (size_t)kSmallCols * ny + (size_t)ny * odd(nx) + (size_t)kSmallCols * odd(nx);
  return 8 * (fwd > back ? fwd : back);
}

}  // namespace

// Line of the dispatch: see kSmallN in slice_transform.h
bool small_plane_f64(const Field& f) { return f.n[0] <= kSmallN && f.n[1] <= kSmallN; }
bool small_z_f64(const Field& f) { return f.n[2] <= kSmallN; }

fdi_status launch_small_plane(fdi_plan* p, const Field& f, bool forward, const double* in, double* out,
                              bool accumulate, bool pdl, const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, forward ? "planes_fwd_f64" : "planes_back_f64", s);
  SmallArgs a{};
  a.in = in;
  a.out = out;
  a.nx = f.n[0];
  a.ny = f.n[1];
  a.Tx = forward ? f.ax[0]->Einv : f.ax[0]->E;
  a.Ty = forward ? f.ax[1]->Einv : f.ax[1]->E;
  a.accumulate = accumulate ? 1 : 0;
  const int groups = ((forward ? a.nx : a.ny) + kSmallCols - 1) / kSmallCols;
  static_assert(8 * (3 * kSmallN * (kSmallN + 1) + 2 * kSmallCols * (kSmallN + 1)) <= 48 * 1024, "shared memory");
  FDI_CUDA_TRY(launch_pdl(pdl && p->pdl, forward ? k_small_forward : k_small_back,
                          dim3((unsigned)groups, (unsigned)f.n[2]), dim3(kSmallThreads), plane_bytes(a.nx, a.ny), s, a,
                          skip));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_small_z(fdi_plan* p, const Field& f, double sigma, double lambda, double* data, const int* skip,
                          cudaStream_t s) {
  FDI_KTIMER(p, "transform_z_f64", s);
  SmallZArgs a{};
  a.data = data;
  a.Tf = f.ax[2]->Einv;
  a.Tb = f.ax[2]->E;
  a.lx = f.ax[0]->lam;
  a.ly = f.ax[1]->lam;
  a.lz = f.ax[2]->lam;
  a.nx = f.n[0];
  a.ny = f.n[1];
  a.nz = f.n[2];
  a.singular = (sigma == 0.0 && f.zero_flux_all) ? 1 : 0;
  a.sigma = sigma;
  a.lambda = lambda;
  const unsigned groups = (unsigned)((a.nx * a.ny + kSmallCols - 1) / kSmallCols);
  const size_t bytes = 8 * ((size_t)2 * a.nz * odd(a.nz) + (size_t)2 * a.nz * kSmallCols);
  FDI_CUDA_TRY(launch_pdl(p->pdl, k_small_z, dim3(groups), dim3(kSmallThreads), bytes, s, a, skip));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

}  // namespace fdi
