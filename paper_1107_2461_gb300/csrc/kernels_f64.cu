// FP64 kernels of the direct Helmholtz / Laplace inverse (the plain FP64 path).
//
//   k_slab_f64    out[b][k][c] = sum_j T_b[k][j] in[b][j][c]  radial transforms of
//                 the cylindrical TPF, one matrix per theta mode (the other
//                 transforms: slice_transform.cu)
//   k_thomas_f64  per (x-mode, y-mode) line the tridiagonal z-system
//                 [(sigma - lam (Lx_i + Ly_j)) M_z - lam K_z] u = M_z f   (TPT,
//                 end of Sec. 3: Thomas algorithm in one direction)
//   k_divide_f64  u_ijk = f_ijk / (sigma - lam (Lx_i + Ly_j + Lz_k))  (Eq. 26-28)
//   k_residual_f64 r = b - A u with the 7-point finite-volume stencil in flux form,
//                 the sums of r^2 and b^2 (per-block partial sums, added by the
//                 block that finishes last in a fixed order) and the convergence
//                 check
//
// GB300 runs FP64 at about 2 FMA/clk/SM, so k_slab_f64 is FP64-pipe bound; it is
// register-tiled (4x4 outputs per thread, 64x64 tiles staged in shared
// memory) so that every shared-memory load feeds two FMAs.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fdi_internal.h"
#include "reduce.cuh"
#include "slice_transform.h"

namespace fdi {
namespace {

constexpr int TB = 64;   // tile edge
constexpr int TK = 16;   // k-chunk
constexpr int kResBlocks = 152 * 8;
constexpr int kResThreads = 256;

// Element (j, c) of the input of batch b at A[b * zin + j * rs + c], of the
// output C[b * zout + k * rs + c]; the matrix of batch b is T + b * tz (tz = 0:
// one matrix for every batch).  A y pass over z-slabs has rs = ncols, zin =
// nin * ncols; a per-mode transform (cylindrical TPF: one radial matrix per
// theta mode) has batch = mode, rs = the row stride of the field, tz = nin * nout.
__global__ void __launch_bounds__(256) k_slab_f64(const double* __restrict__ A, double* __restrict__ C,
                                                  const double* __restrict__ T, int nin, int nout,
                                                  long long ncols, long long rs, long long zin, long long zout,
                                                  long long tz, const int* __restrict__ skip) {
  if (skip && *skip) return;
  __shared__ double As[TK][TB + 1];  // T tile [j][k]
  __shared__ double Bs[TK][TB + 1];  // data tile [j][c]
  const long long b = blockIdx.z;
  A += b * zin;
  C += b * zout;
  T += b * tz;
  const long long c0 = (long long)blockIdx.x * TB;
  const int k0 = blockIdx.y * TB;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[a][q] = 0.0;
  for (int j0 = 0; j0 < nin; j0 += TK) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int jj = threadIdx.x % TK, kk = threadIdx.x / TK + 16 * r;
      int j = j0 + jj, k = k0 + kk;
      As[jj][kk] = (k < nout && j < nin) ? T[(long long)k * nin + j] : 0.0;
      int cc = threadIdx.x % TB, jr = threadIdx.x / TB + 4 * r;
      long long col = c0 + cc;
      int j2 = j0 + jr;
      Bs[jr][cc] = (col < ncols && j2 < nin) ? A[(long long)j2 * rs + col] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int jj = 0; jj < TK; ++jj) {
      double a[4], bb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = As[jj][ty + 16 * q];
        bb[q] = Bs[jj][tx + 16 * q];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[q][c] = fma(a[q], bb[c], acc[q][c]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int k = k0 + ty + 16 * q;
    if (k >= nout) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      long long col = c0 + tx + 16 * c;
      if (col < ncols) C[(long long)k * rs + col] = acc[q][c];
    }
  }
}

// Thomas sweep along z (TPT, end of Sec. 3) in FP64 for every (x-mode,
// y-mode) line: [(sigma - lam Lx_i) M_z - lam K_z - lam Ly_j W] u = M_z f with
// W = M_z (Cartesian) or the theta weight A g (cylindrical plans).  The line
// factorisation (c'_k and the reciprocal pivots) depends on (sigma, lambda,
// field) only; it is kept in a per-workspace cache whose key the sweep reads
// on the device: a matching key runs the cached sweep (about four FP64
// operations per point, no divide), any other runs the factorising sweep and
// refreshes the cache (the key is written by the sweep's last block to finish, so
// every block of a sweep sees the same key, also in replayed graphs).  T is
// the field type: double (FP64 path) or float (the mixed path's FP32 fields,
// configuration 4, FP64 recurrence).  Field element (k, line l) at
// k * kstride + (l / ny) * pitch + l % ny, l = i * ny + j ... for the FP64
// path pitch = ny = lines per x mode is replaced by the [z][y][x] order below.
struct ThomasArgs {
  const void* in;
  void* out;
  double* cs;        // scratch c'_k (no cache)
  int nx, ny, nz;
  int mixed_layout;  // 0: FP64 field [z][y][x] (line l = j*nx + i); 1: FP32 [z][i][pitch] (l = i*ny + j)
  int pitch;
  long long kstride;
  const double* lamx;
  const double* lamy;
  const double* mz;
  const double* kdz;
  const double* koz;
  const double* wy;  // per z: weight of the y eigenvalue (cylindrical theta: A_i g_i); null: M_z
  double sigma, lambda;
  int field;
  int singular_possible;  // sigma == 0 and zero-flux walls everywhere
  double* cinv;      // factor cache: reciprocal pivots [k][line] (null: no cache)
  double* ccp;       //               c'_k [k][line]
  double* key;       //               (sigma, lambda, field) of the cached factors
  unsigned* ticket;  // counts finished blocks (zero between launches)
  long long q;       // line points per plane of the cache (>= lines)
  float* fmax;       // FP32 fields: atomic max |u| (the next pass's scale)
};

__device__ __forceinline__ void warp_max_out(float v, float* fmax) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v > 0.f) atomicMax(reinterpret_cast<unsigned int*>(fmax), __float_as_uint(v));
}

// kTP planes per block of loads: every sweep reads its next block before it
// computes the current one, so a step does not wait for memory (between events,
// 64^3: 41 us with one step's loads in flight, 24 us in blocks of 8 or 16; 128^3:
// 136, 57 and 47 us).  Single-warp blocks take 16; large fields keep 8, whose
// registers leave enough warps per SM to stream 40 bytes per point (256^3 solve
// 1.95 ms before, 1.82 with 8, 1.90 with 16).

// The singular line of the zero-flux Laplacian (Eq. 28 reading), by a block of
// its own: project the right-hand side to zero M_z-weighted mean, pin u_0 = 0,
// solve rows 1 .. nz-1, remove the weighted mean of the solution.  The line is
// staged in shared memory; the sums and copies run over the block's threads, the
// recurrences in one.
template <typename T>
__device__ void thomas_singular_line(const ThomasArgs& a, const double* s_m, const double* s_lo, const T* in, T* out,
                                     bool cached, float& vmax) {
  __shared__ double s_f[kMaxN], s_c[kMaxN], s_i[kMaxN];
  __shared__ double s_sum[2];
  const int nz = a.nz, t = threadIdx.x;
  for (int k = t; k < nz; k += blockDim.x) {
    s_f[k] = (double)in[k * a.kstride];
    if (cached) {
      s_i[k] = a.cinv[k * a.q];
      s_c[k] = a.ccp[k * a.q];
    }
  }
  __syncthreads();
  auto weighted = [&]() {  // (sum M, sum M s_f) by the first warp
    if (t < 32) {
      double sm = 0.0, sf = 0.0;
      for (int k = t; k < nz; k += 32) {
        sm += s_m[k];
        sf = fma(s_m[k], s_f[k], sf);
      }
      const double v = red::warp_sum2(sm, sf);
      if (t == 0) s_sum[0] = v;
      if (t == 16) s_sum[1] = v;
    }
    __syncthreads();
    return s_sum[1] / s_sum[0];
  };
  const double mu = weighted();
  if (t == 0) {
    double cprev = 0.0, dprev = 0.0;
    for (int k = 1; k < nz; ++k) {
      const double lo = (k > 1) ? -s_lo[k - 1] : 0.0;
      double inv;
      if (cached) {
        inv = s_i[k];
      } else {
        const double up = (k + 1 < nz) ? -s_lo[k] : 0.0;
        inv = 1.0 / (-a.lambda * a.kdz[k] - lo * cprev);
        cprev = up * inv;
        s_i[k] = inv;
        s_c[k] = cprev;
      }
      dprev = (s_m[k] * (s_f[k] - mu) - lo * dprev) * inv;
      s_f[k] = dprev;
    }
    double u = dprev;
    for (int k = nz - 2; k >= 1; --k) {
      u = s_f[k] - s_c[k] * u;
      s_f[k] = u;
    }
    s_f[0] = 0.0;
  }
  __syncthreads();
  const double mean = weighted();
  for (int k = t; k < nz; k += blockDim.x) {
    const double w = s_f[k] - mean;
    out[k * a.kstride] = (T)w;
    vmax = fmaxf(vmax, fabsf((float)w));
    if (a.cinv && !cached) {
      a.cinv[k * a.q] = s_i[k];
      a.ccp[k * a.q] = s_c[k];
    }
  }
}

template <typename T, int kTP>
__global__ void __launch_bounds__(128) k_thomas_f64(ThomasArgs a, const int* __restrict__ skip) {
  __shared__ double s_m[kMaxN], s_lo[kMaxN], s_kd[kMaxN];  // M_k, lambda K_{k,k+1}, lambda Kd_k
  const int nz = a.nz;
  for (int k = threadIdx.x; k < nz; k += blockDim.x) {
    s_m[k] = a.mz[k];
    s_lo[k] = a.lambda * a.koz[k];
    s_kd[k] = a.lambda * a.kdz[k];
  }
  __syncthreads();
  pdl_wait();  // (the coefficients are plan data)
  if (skip && *skip) return;
  const long long NL = (long long)a.nx * a.ny;
  // a singular problem has one block more, which solves the null line (0, 0)
  const bool null_block = a.singular_possible && blockIdx.x == gridDim.x - 1;
  const long long l0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  // (the scale of the mixed path; the conversion would take the FP64 pipe's time)
  constexpr bool kMax = std::is_same<T, float>::value;
  float vmax = 0.f;
  const long long l = null_block ? 0 : (l0 < NL ? l0 : NL - 1);
  const bool live = !null_block && l0 < NL && !(a.singular_possible && l0 == 0);
  int i, j;
  long long off;
  if (a.mixed_layout) {
    i = (int)(l / a.ny);
    j = (int)(l % a.ny);
    off = (long long)i * a.pitch + j;
  } else {
    i = (int)(l % a.nx);
    j = (int)(l / a.nx);
    off = l;
  }
  const T* in = static_cast<const T*>(a.in) + off;
  T* out = static_cast<T*>(a.out) + off;
  const long long ks = a.kstride;
  const bool cached = a.cinv && a.key[0] == a.sigma && a.key[1] == a.lambda && a.key[2] == (double)a.field;
  if (null_block) {
    thomas_singular_line<T>(a, s_m, s_lo, in, out, cached, vmax);
  } else if (live) {
    const double lab = a.lamx[i] + a.lamy[j];
    // the y eigenvalue takes its own weight on cylindrical plans (Eq. 44: the
    // theta eigenvalue multiplies the discrete 1/r^2 of the radial cell)
    const double s = a.sigma - a.lambda * (a.wy ? a.lamx[i] : lab);
    const double ly = a.wy ? a.lambda * a.lamy[j] : 0.0;
    double* cp_arr = a.cinv ? a.ccp + l : a.cs + off;
    const long long cstride = a.cinv ? a.q : ks;
    const double* inv_arr = a.cinv + l;
    T f[kTP], fn[kTP];
    double iv[kTP], ivn[kTP];
    auto load_fwd = [&](int k0, T (&x)[kTP], double (&y)[kTP]) {
#pragma unroll
      for (int u = 0; u < kTP; ++u) {
        const int k = min(k0 + u, nz - 1);
        x[u] = in[k * ks];
        if (cached) y[u] = inv_arr[k * a.q];
      }
    };
    double d = 0.0;
    load_fwd(0, f, iv);
    if (cached) {
      for (int k0 = 0; k0 < nz; k0 += kTP) {
        if (k0 + kTP < nz) load_fwd(k0 + kTP, fn, ivn);
#pragma unroll
        for (int u = 0; u < kTP; ++u) {
          const int k = k0 + u;
          if (k < nz) {
            double t = __dmul_rn(s_m[k], (double)f[u]);
            if (k > 0) t = __fma_rn(s_lo[k - 1], d, t);
            d = __dmul_rn(t, iv[u]);
            out[k * ks] = (T)d;
          }
          f[u] = fn[u];
          iv[u] = ivn[u];
        }
      }
    } else {
      double cprev = 0.0;
      for (int k0 = 0; k0 < nz; k0 += kTP) {
        if (k0 + kTP < nz) load_fwd(k0 + kTP, fn, ivn);
#pragma unroll 1
        for (int u = 0; u < kTP; ++u) {
          const int k = k0 + u;
          if (k >= nz) break;
          const double lo = (k > 0) ? -s_lo[k - 1] : 0.0;
          const double up = (k + 1 < nz) ? -s_lo[k] : 0.0;
          double di = s * s_m[k] - s_kd[k];
          if (a.wy) di -= ly * a.wy[k];
          const double inv = 1.0 / (di - lo * cprev);
          cprev = up * inv;
          // the same operations, in the same order, as the cached sweep: a
          // solve gives the same bits whether its factors were cached or not
          double t = __dmul_rn(s_m[k], (double)f[0]);
          if (k > 0) t = __fma_rn(s_lo[k - 1], d, t);
          d = __dmul_rn(t, inv);
          cp_arr[k * cstride] = cprev;
          if (a.cinv) a.cinv[l + k * a.q] = inv;
          out[k * ks] = (T)d;
#pragma unroll
          for (int q = 0; q + 1 < kTP; ++q) f[q] = f[q + 1];
        }
#pragma unroll
        for (int u = 0; u < kTP; ++u) f[u] = fn[u];
      }
    }
    // back substitution, blocks from the top: f holds d', iv holds c'
    auto load_back = [&](int k0, T (&x)[kTP], double (&y)[kTP]) {
#pragma unroll
      for (int u = 0; u < kTP; ++u) {
        const int k = max(k0 - u, 0);
        x[u] = out[k * ks];
        y[u] = cp_arr[k * cstride];
      }
    };
    double u_ = d;
    if (kMax) vmax = fmaxf(vmax, fabsf((float)u_));
    load_back(nz - 2, f, iv);
    for (int k0 = nz - 2; k0 >= 0; k0 -= kTP) {
      if (k0 - kTP >= 0) load_back(k0 - kTP, fn, ivn);
#pragma unroll
      for (int u = 0; u < kTP; ++u) {
        const int k = k0 - u;
        if (k >= 0) {
          u_ = __fma_rn(-iv[u], u_, (double)f[u]);
          out[k * ks] = (T)u_;
          if (kMax) vmax = fmaxf(vmax, fabsf((float)u_));
        }
        f[u] = fn[u];
        iv[u] = ivn[u];
      }
    }
  }
  // one reduction point for the whole warp
  if (kMax && a.fmax) warp_max_out(vmax, a.fmax);
  if (a.cinv) {
    // the last block to finish records whose factors the cache holds now: every
    // block has read the old key by then
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(a.ticket, 1u) == gridDim.x - 1) {
        a.key[0] = a.sigma;
        a.key[1] = a.lambda;
        a.key[2] = (double)a.field;
        *a.ticket = 0u;
      }
    }
  }
}

// threads per block: single warps while that still leaves SM quarters idle.  Whole
// solves, single warps of 16 planes against 128 threads of 8 (us): 128 x 128 x 128
// 241 / 247, 140 x 140 x 128 386 / 398, 192 x 192 x 128 581 / 589, 224 x 224 x 128
// 1442 / 1456, 256 x 256 x 128 1814 / 1773: the line could lie as far up as 50
// thousand lines, for 1 to 3%.
int thomas_threads(long long lines) { return lines <= 152 * 128 ? 32 : 128; }

__global__ void k_divide_f64(double* __restrict__ data, int nx, int ny, int nz, const double* __restrict__ lx,
                             const double* __restrict__ ly, const double* __restrict__ lz, double sigma,
                             double lambda, int singular_possible, const int* __restrict__ skip) {
  pdl_wait();
  if (skip && *skip) return;
  const long long P = (long long)nx * ny * nz;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (long long)gridDim.x * blockDim.x) {
    int i = (int)(p % nx);
    long long t = p / nx;
    int j = (int)(t % ny), k = (int)(t / ny);
    double ls = lx[i] + ly[j] + lz[k];
    double dv = sigma - lambda * ls;
    data[p] = (singular_possible && ls == 0.0) ? 0.0 : data[p] / dv;
  }
}

// cylindrical TPF (Eq. 46): data [k][j][i] with k the radial mode of theta
// mode j; u /= sigma - lam (Lx_i + Lr_{j,k})
__global__ void k_divide_modes_f64(double* __restrict__ data, int nx, int ny, int nz, const double* __restrict__ lx,
                                   const double* __restrict__ lr, double sigma, double lambda,
                                   const int* __restrict__ skip) {
  if (skip && *skip) return;
  const long long P = (long long)nx * ny * nz;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(p % nx);
    const long long t = p / nx;
    const int j = (int)(t % ny), k = (int)(t / ny);
    data[p] = data[p] / (sigma - lambda * (lx[i] + lr[(long long)j * nz + k]));
  }
}

// Residual r = b - sigma u + lambda L u (7-point flux form) and ||r||^2, ||b||^2.
// FP64 arithmetic bounds it: 2 lane-operations per clock and SM, so the form
// below counts them.  A block of 256 threads covers 64 x 8 columns and marches
// over up to kResZ planes; a thread owns columns i and i + 32 of one row.  The
// lambda-scaled weights are formed once per thread (x, y) or block (z); a
// Dirichlet wall is a neighbour of value zero with the wall's weight, a zero-flux
// wall one of weight zero, so no cell needs an extra term or a branch; the z
// difference is shared by two planes and the x difference by two columns (a
// shuffle moves it to the next lane, only lane 0 forms its own).  13.5
// operations per point instead of 22: 256^3 0.72 to 0.48 ms, and the block
// that finishes last reduces the partial sums (no second launch).
constexpr int kResZ = 8;

struct ResidF64 {
  int nx, ny, nz, zchunk;
  const double* wp[3];
  const double* wm[3];
  const double* w0[3];
  const double* wyk;  // periodic y with the flux weight wyk[k] of plane k (cylindrical theta)
  const double* b;
  const double* u;
  double* r;
  double sigma, lambda, tol;
  DevStatus* st;
  int sub_mean, first;
  double* partials;
  unsigned* ticket;
  cudaGraphConditionalHandle next_round;  // captured solves: the next refinement round's condition
};

__device__ void finish_residual(const ResidF64& a, double rr, double bb) {
  DevStatus* st = a.st;
  if (a.first) {  // the solve's status starts here
    st->tol_used = a.tol;
    st->iters = 0;
    st->error = 0;
    st->refine_steps = 0;
    st->bnorm2 = bb;
  } else {
    st->refine_steps += 1;
    bb = st->bnorm2;
  }
  const double rel = (bb > 0.0) ? sqrt(rr / bb) : sqrt(rr);
  st->rel_res = rel;
  if (a.first && !isfinite(bb)) {
    st->error = 7;  // non-finite right-hand side
    st->done = 1;
  } else if (!isfinite(rel)) {
    st->error = 1;
    st->done = 1;
  } else {
    st->done = rel <= a.tol ? 1 : 0;
  }
  if (a.next_round) cudaGraphSetConditional(a.next_round, st->done ? 0u : 1u);
}

template <int SIG, bool CYL, bool FIRST>
__global__ void __launch_bounds__(kResThreads, 2) k_residual_f64(const ResidF64 a, const int* __restrict__ skip) {
  pdl_wait();
  if (skip && *skip) return;
  __shared__ double sh[32];
  __shared__ double s_wz[3][kResZ];
  __shared__ int s_last;
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
  const int k0 = blockIdx.z * a.zchunk, k1 = min(nz, k0 + a.zchunk);
  if (threadIdx.x < k1 - k0) {
    const int q = threadIdx.x, k = k0 + q;
    s_wz[0][q] = a.lambda * (k == nz - 1 ? -a.w0[2][k] : a.wp[2][k]);
    s_wz[1][q] = -a.lambda * (k == 0 ? -a.w0[2][k] : a.wm[2][k]);
    s_wz[2][q] = CYL ? a.lambda * a.wyk[k] : 0.0;
  }
  const int iA = blockIdx.x * 64 + lane, iB = iA + 32, j = blockIdx.y * 8 + wy;
  const bool actA = j < ny && iA < nx, actB = j < ny && iB < nx;
  const int ca = min(iA, nx - 1), cb = min(iB, nx - 1), jc = min(j, ny - 1);
  const bool eA = ca == nx - 1, eB = cb == nx - 1, wA = ca == 0;  // next to an x wall
  const double wpA = a.lambda * (eA ? -a.w0[0][ca] : a.wp[0][ca]);
  const double wpB = a.lambda * (eB ? -a.w0[0][cb] : a.wp[0][cb]);
  const double wmA = -a.lambda * (wA ? -a.w0[0][ca] : a.wm[0][ca]);
  const double wmB = -a.lambda * a.wm[0][cb];  // column B is never the first
  double wpy = 0.0, wmy = 0.0;
  if (!CYL) {
    wpy = a.lambda * (jc == ny - 1 ? -a.w0[1][jc] : a.wp[1][jc]);
    wmy = a.lambda * (jc == 0 ? -a.w0[1][jc] : a.wm[1][jc]);
  }
  const bool gN = !CYL && jc == ny - 1, gS = !CYL && jc == 0;  // zero neighbours
  const long long pl = (long long)nx * ny;
  const long long rowc = (long long)jc * nx;
  const long long rown = (long long)(jc + 1 < ny ? jc + 1 : (CYL ? 0 : jc)) * nx;
  const long long rows = (long long)(jc > 0 ? jc - 1 : (CYL ? ny - 1 : jc)) * nx;
  // lane 31 reads the column east of the block's, lane 0 the one west of it
  const int ce = lane == 31 ? min(iB + 1, nx - 1) : max(iA - 1, 0);
  const double mb = a.sub_mean ? a.st->mean_b : 0.0;
  const double* u = a.u + k0 * pl;
  const double* bp = a.b + k0 * pl + rowc;
  double* rp = a.r + k0 * pl + rowc;
  double CA = u[rowc + ca], CB = u[rowc + cb];
  double dA, dB;  // u_k - u_{k-1}
  {
    const double MA = k0 > 0 ? u[rowc + ca - pl] : 0.0, MB = k0 > 0 ? u[rowc + cb - pl] : 0.0;
    dA = CA - MA;
    dB = CB - MB;
  }
  double srr = 0.0, sbb = 0.0;
  __syncthreads();
  for (int q = 0; q < k1 - k0; ++q) {
    const bool top = k0 + q == nz - 1;
    double PA = 0.0, PB = 0.0;
    if (!top) {
      PA = u[pl + rowc + ca];
      PB = u[pl + rowc + cb];
    }
    const double NA = gN ? 0.0 : u[rown + ca], NB = gN ? 0.0 : u[rown + cb];
    const double SA = gS ? 0.0 : u[rows + ca], SB = gS ? 0.0 : u[rows + cb];
    double E = u[rowc + ce];
    double accA = bp[ca], accB = bp[cb];
    const double wpz = s_wz[0][q], wmz = s_wz[1][q];
    if (CYL) wpy = wmy = s_wz[2][q];
    if (a.sub_mean) {
      accA -= mb;
      accB -= mb;
    }
    if (FIRST) {
      sbb = fma(actA ? accA : 0.0, accA, sbb);
      sbb = fma(actB ? accB : 0.0, accB, sbb);
    }
    // x: differences to the east, moved one lane up for the west faces
    const double rA = __shfl_sync(0xffffffffu, CA, (lane + 1) & 31), rB = __shfl_sync(0xffffffffu, CB, (lane + 1) & 31);
    double eastA = lane == 31 ? rB : rA, eastB = lane == 31 ? E : rB;
    if (eA) eastA = 0.0;
    if (eB) eastB = 0.0;
    const double xA = eastA - CA, xB = eastB - CB;
    if (wA) E = 0.0;
    const double own = CA - E;  // lane 0's west difference
    const double vA = __shfl_sync(0xffffffffu, xA, (lane + 31) & 31), vB = __shfl_sync(0xffffffffu, xB, (lane + 31) & 31);
    const double westA = lane == 0 ? own : vA, westB = lane == 0 ? vA : vB;
    if (SIG == 1) {
      accA -= CA;
      accB -= CB;
    } else if (SIG == 2) {
      accA = fma(-a.sigma, CA, accA);
      accB = fma(-a.sigma, CB, accB);
    }
    const double uA = PA - CA, uB = PB - CB;
    accA = fma(wpA, xA, accA);
    accB = fma(wpB, xB, accB);
    accA = fma(wmA, westA, accA);
    accB = fma(wmB, westB, accB);
    accA = fma(wpy, NA - CA, accA);
    accB = fma(wpy, NB - CB, accB);
    accA = fma(wmy, SA - CA, accA);
    accB = fma(wmy, SB - CB, accB);
    accA = fma(wpz, uA, accA);
    accB = fma(wpz, uB, accB);
    accA = fma(wmz, dA, accA);
    accB = fma(wmz, dB, accB);
    srr = fma(actA ? accA : 0.0, accA, srr);
    srr = fma(actB ? accB : 0.0, accB, srr);
    if (actA) rp[ca] = accA;
    if (actB) rp[cb] = accB;
    CA = PA;
    CB = PB;
    dA = uA;
    dB = uB;
    u += pl;
    bp += pl;
    rp += pl;
  }
  red::block_sum2(srr, sbb, kResThreads / 32, sh);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  const unsigned bid = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) {
    reinterpret_cast<double2*>(a.partials)[bid] = make_double2(srr, sbb);
    __threadfence();
    s_last = atomicAdd(a.ticket, 1u) == nb - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double x = 0.0, y = 0.0;
  for (unsigned q = threadIdx.x; q < nb; q += kResThreads) {
    const double2 v = reinterpret_cast<const double2*>(a.partials)[q];
    x += v.x;
    if (FIRST) y += v.y;
  }
  red::block_sum2(x, y, (int)min((unsigned)(kResThreads / 32), (nb + 31) / 32), sh);
  if (threadIdx.x == 0) {
    *a.ticket = 0u;
    finish_residual(a, x, y);
  }
}

// Volume-weighted mean of b (zero-flux Laplace problem): one warp per x line,
// one FP64 multiply-add per value; the last block divides by the sum of volumes.
__global__ void __launch_bounds__(kResThreads) k_vmean(const double* __restrict__ b, int nx, int ny, int nz,
                                                       const double* __restrict__ mx, const double* __restrict__ my,
                                                       const double* __restrict__ mz, double vol_sum,
                                                       double* __restrict__ partials, unsigned* ticket, DevStatus* st) {
  pdl_wait();
  __shared__ double sh[32];
  __shared__ int s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s = 0.0, zero = 0.0;
  for (int l = blockIdx.x * (kResThreads / 32) + warp; l < ny * nz; l += gridDim.x * (kResThreads / 32)) {
    const double* row = b + (long long)l * nx;
    double t = 0.0;
    for (int i = lane; i < nx; i += 32) t = fma(mx[i], row[i], t);
    s = fma(my[l % ny] * mz[l / ny], t, s);
  }
  red::block_sum2(s, zero, kResThreads / 32, sh);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  s = zero = 0.0;
  for (unsigned q = threadIdx.x; q < gridDim.x; q += kResThreads) s += partials[q];
  red::block_sum2(s, zero, (int)min((unsigned)(kResThreads / 32), (gridDim.x + 31) / 32), sh);
  if (threadIdx.x == 0) {
    *ticket = 0u;
    st->mean_b = s / vol_sum;
  }
}

template <bool CYL>
void (*residual_kernel(double sigma, bool first))(const ResidF64, const int*) {
  if (sigma == 0.0) return first ? k_residual_f64<0, CYL, true> : k_residual_f64<0, CYL, false>;
  if (sigma == 1.0) return first ? k_residual_f64<1, CYL, true> : k_residual_f64<1, CYL, false>;
  return first ? k_residual_f64<2, CYL, true> : k_residual_f64<2, CYL, false>;
}

}  // namespace

fdi_status launch_axis_f64(fdi_plan* p, const Field& f, int d, bool forward, const double* in, double* out,
                           bool accumulate, bool pdl, const int* skip, cudaStream_t s) {
  const Axis* ax = f.ax[d];
  const long long nx = f.n[0], ny = f.n[1];
  FDI_KTIMER(p, d == 0 ? "transform_x_f64" : (d == 1 ? "transform_y_f64" : "transform_z_f64"), s);
  const SliceAxis* sa = static_cast<const SliceAxis*>(ax->slices);
  if (!sa) {
    set_error("direction has no FP64 transform");
    return FDI_ERR_INVALID_ARG;
  }
  SliceLines g;
  g.R = f.P / ax->n;
  if (d == 0) {  // x lines: rows (z, y)
    g.S = g.R;
    g.rs = nx;
    g.ks = 1;
  } else if (d == 1) {  // y lines: (z, x)
    g.S = nx;
    g.slab = nx * ny;
    g.rs = 1;
    g.ks = nx;
  } else {  // z lines: (y, x)
    g.S = nx * ny;
    g.rs = 1;
    g.ks = nx * ny;
  }
  return launch_slice_transform(p, forward ? sa->fwd : sa->bwd, in, out, g, accumulate, pdl, skip, s);
}

fdi_status launch_modes_f64(fdi_plan* p, const double* in, double* out, const double* T_all, int n, int nx,
                            int ny, const int* skip, cudaStream_t s) {
  // field [n][ny][nx]; for every y index j (a theta mode) the n x n matrix
  // T_all + j n^2 contracts the outer index
  FDI_KTIMER(p, "transform_r_modes_f64", s);
  dim3 grid((unsigned)((nx + TB - 1) / TB), (unsigned)((n + TB - 1) / TB), (unsigned)ny);
  k_slab_f64<<<grid, 256, 0, s>>>(in, out, T_all, n, n, nx, (long long)nx * ny, nx, nx, (long long)n * n, skip);
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_thomas_f64(fdi_plan* p, const Field& f, double sigma, double lambda, int field, const double* in,
                             double* out, double* scratch, const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, "thomas_z_f64", s);
  ThomasArgs a{};
  a.in = in;
  a.out = out;
  a.cs = scratch;
  a.nx = f.n[0];
  a.ny = f.n[1];
  a.nz = f.n[2];
  a.mixed_layout = 0;
  a.pitch = f.n[0];
  a.kstride = (long long)f.n[0] * f.n[1];
  a.lamx = f.ax[0]->lam;
  a.lamy = f.ax[1]->lam;
  a.mz = f.ax[2]->m;
  a.kdz = f.ax[2]->kd;
  a.koz = f.ax[2]->ko;
  a.wy = p->cyl_wy;
  a.sigma = sigma;
  a.lambda = lambda;
  a.field = field;
  a.singular_possible = (sigma == 0.0 && f.zero_flux_all) ? 1 : 0;
  const long long NL = (long long)a.nx * a.ny;
  const bool cache = p->tf && p->tf_q >= f.P;
  if (cache) {
    a.q = NL;
    a.cinv = p->tf;
    a.ccp = p->tf + p->tf_q;
    a.key = p->tf + 2 * p->tf_q;
    a.ticket = p->d_counter + 1;
  }
  const int nt = thomas_threads(NL);
  FDI_CUDA_TRY(launch_pdl(p->pdl, nt == 32 ? k_thomas_f64<double, 16> : k_thomas_f64<double, 8>, dim3((unsigned)((NL + nt - 1) / nt) + a.singular_possible),
                          dim3(nt), 0, s, a, skip));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_thomas_cached_f32(fdi_plan* p, const Field& f, double sigma, double lambda, int field, float* data,
                                    int pitch, long long plane, float* fmax, const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, "thomas_z_f64rec", s);
  ThomasArgs a{};
  a.in = data;
  a.out = data;
  a.cs = nullptr;
  a.nx = f.n[0];
  a.ny = f.n[1];
  a.nz = f.n[2];
  a.mixed_layout = 1;
  a.pitch = pitch;
  a.kstride = plane;
  a.lamx = f.ax[0]->lam;
  a.lamy = f.ax[1]->lam;
  a.mz = f.ax[2]->m;
  a.kdz = f.ax[2]->kd;
  a.koz = f.ax[2]->ko;
  a.wy = p->cyl_wy;
  a.sigma = sigma;
  a.lambda = lambda;
  a.field = field;
  a.singular_possible = 0;  // the singular problem keeps the FP32 sweep's null-line kernel
  a.fmax = fmax;
  const long long NL = (long long)a.nx * a.ny;
  a.q = NL;
  a.cinv = p->tf;
  a.ccp = p->tf + p->tf_q;
  a.key = p->tf + 2 * p->tf_q;
  a.ticket = p->d_counter + 1;
  const int nt = thomas_threads(NL);
  if (nt == 32)
    k_thomas_f64<float, 16><<<(unsigned)((NL + nt - 1) / nt), nt, 0, s>>>(a, skip);
  else
    k_thomas_f64<float, 8><<<(unsigned)((NL + nt - 1) / nt), nt, 0, s>>>(a, skip);
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_divide_f64(fdi_plan* p, const Field& f, double sigma, double lambda, double* data,
                             const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, "divide_f64", s);
  int sp = (sigma == 0.0 && f.zero_flux_all) ? 1 : 0;
  const unsigned blocks = (unsigned)std::min<long long>(152 * 8, (f.P + 255) / 256);
  FDI_CUDA_TRY(launch_pdl(p->pdl, k_divide_f64, dim3(blocks), dim3(256), 0, s, data, f.n[0], f.n[1], f.n[2],
                          (const double*)f.ax[0]->lam, (const double*)f.ax[1]->lam, (const double*)f.ax[2]->lam, sigma,
                          lambda, sp, skip));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_divide_modes_f64(fdi_plan* p, const Field& f, double sigma, double lambda, double* data,
                                  const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, "divide_f64", s);
  k_divide_modes_f64<<<152 * 8, 256, 0, s>>>(data, f.n[0], f.n[1], f.n[2], f.ax[0]->lam, p->cyl_lr, sigma, lambda,
                                            skip);
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_residual_f64(fdi_plan* p, const Field& f, double sigma, double lambda, const double* b,
                               const double* u, double* r, bool subtract_mean, bool first,
                               cudaGraphConditionalHandle next_round, const int* skip, cudaStream_t s) {
  FDI_KTIMER(p, "residual_f64", s);
  ResidF64 a{};
  a.nx = f.n[0];
  a.ny = f.n[1];
  a.nz = f.n[2];
  for (int d = 0; d < 3; ++d) {
    a.wp[d] = f.ax[d]->wp;
    a.wm[d] = f.ax[d]->wm;
    a.w0[d] = f.ax[d]->w0;
  }
  a.wyk = p->cyl_wres;
  a.b = b;
  a.u = u;
  a.r = r;
  a.sigma = sigma;
  a.lambda = lambda;
  a.tol = p->tol;
  a.st = p->d_status;
  a.sub_mean = subtract_mean ? 1 : 0;
  a.first = first ? 1 : 0;
  a.partials = p->partials;
  a.ticket = p->d_counter;
  a.next_round = next_round;
  // the march length with the least work on the busiest SM, a march costing its
  // planes and about one plane's time for its start (a whole FP64 solve with 8, the
  // longest, and with the rule's length: 64^3 86 and 78 us, 80^3 133 and 125, 112^3
  // 214 and 209, 128^3 246 and 238; from 48^3 to 256^3 no other length was faster)
  const dim3 cols((unsigned)((a.nx + 63) / 64), (unsigned)((a.ny + 7) / 8));
  auto blocks = [&](int zc) { return (long long)cols.x * cols.y * ((a.nz + zc - 1) / zc); };
  auto cost = [&](int zc) { return (blocks(zc) + 151) / 152 * (zc + 1); };
  a.zchunk = kResZ;
  for (int zc = kResZ - 1; zc >= 1; --zc)
    if (cost(zc) < cost(a.zchunk) && blocks(zc) <= p->npartials) a.zchunk = zc;
  const dim3 grid(cols.x, cols.y, (unsigned)((a.nz + a.zchunk - 1) / a.zchunk));
  if ((long long)grid.x * grid.y * grid.z > p->npartials) {
    set_error("grid too large for the reduction buffer");
    return FDI_ERR_INVALID_ARG;
  }
  FDI_CUDA_TRY(launch_pdl(p->pdl, p->cyl_wres ? residual_kernel<true>(sigma, first) : residual_kernel<false>(sigma, first),
                          grid, dim3(kResThreads), 0, s, a, skip));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

fdi_status launch_mean_f64(fdi_plan* p, const Field& f, const double* b, cudaStream_t s) {
  FDI_KTIMER(p, "mean_f64", s);
  const int blocks = std::min(kResBlocks, (f.n[1] * f.n[2] + 15) / 16);
  k_vmean<<<std::max(1, blocks), kResThreads, 0, s>>>(b, f.n[0], f.n[1], f.n[2], f.ax[0]->m, f.ax[1]->m, f.ax[2]->m,
                                                      f.vol_sum, p->partials, p->d_counter, p->d_status);
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

}  // namespace fdi
