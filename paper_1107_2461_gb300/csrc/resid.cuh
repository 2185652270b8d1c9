// Double-float residual of the mixed-precision solve (flux form of Eq. 23)
// and the fixed-order reduction behind its convergence check; shared by the
// pass-by-pass solve (mixed.cu) and the resident small-grid solve
// (resident.cu).
#pragma once
#include <cuda_runtime.h>

#include "df.cuh"
#include "fdi_internal.h"
#include "reduce.cuh"

namespace fdi {
namespace {

// fused final reduction (see finish_if_last)
struct FinishArgs {
  unsigned* counter;    // zero between launches
  const double* partials;
  DevStatus* st;
  double tol;
  int kind, want_mean;
  // captured solves: condition of the next refinement round's graph node
  // (set to "not converged"); 0 when running eagerly
  cudaGraphConditionalHandle next_round = 0;
  // kind 0: where the maximum of the records' first component (max |b|) goes
  float* max_out = nullptr;
};

struct ResidArgs {
  int nx, ny, nz;
  const float2* wp[3];
  const float2* wm[3];
  const float2* w0[3];
  const float2* m[3];
  const float2* wy;     // periodic-y plans: lambda-scaled y flux weight per plane (null otherwise)
  double fast_limit;    // MODE 1: plain FP32 body when ||r_1|| / ||b|| <= fast_limit (0: never)
  float2 sigma, lambda;
  int sig_mode;         // 0: sigma = 0, 1: sigma = 1, 2: general sigma
  const double* b;
  const float* xh;      // solution planes: H, L (= Lh) and the low plane of L
  const float* xl;
  const float* xll;
  const float* r1;      // r_1 as a double-float pair of planes (MODE 1 input)
  const float* r1_lo;
  float* r;             // FP32 residual (the next solve's input)
  float* r_lo;          // MODE 0: low plane of r_1
  int r_pitch;
  int zchunk;           // planes per block (resid_grid)
  double* out;          // FP64 solution output (null: not written)
  float* rmax;          // atomic max |r|
  const DevStatus* st;
  int sub_mean;
  int want_mean;        // accumulate sum V b and sum V (first pass) or sum V x (later passes)
  double* partials;     // per block: sum r^2, sum b^2, sum V b (or V x), sum V
  FinishArgs fin;
};


__device__ __forceinline__ df::F2 ld2(const float2* p) {
  float2 v = *p;
  return df::make(v.x, v.y);
}

// z-marching residual: a block of 32 (x) x 8 (y) threads covers 64 x 8
// columns; each thread a pair of x-neighbours (i0, i0 + 1) of one row j, over a
// range of planes.  Per plane a thread holds its pair at planes k and k + 1 and
// the pairs of rows j - 1 and j + 1 at plane k (the loads of the next plane
// are issued before the current one is computed; with VEC one 8-byte access
// per pair); the x face inside the pair is differenced once for both points,
// the z face below is the previous plane's upper face, and the x neighbours
// outside the pair come from the neighbouring lanes.  Walls need no branch:
// the flux weights are zero across a wall and the clamped neighbour index
// gives an exact zero difference there; only the Dirichlet wall term (nonzero
// next to a wall) is added under a per-thread flag.  Work per block is fixed,
// so the reduction order is too.
//
// Arithmetic: x = xh + xl (double-float).  With the flux weights already
// multiplied by lambda (w' = lambda w, double-float), lambda L x = L'xh + L'xl;
// each flux of L'xh is formed exactly (two-difference of the float values,
// FMA two-product with the weight's high part) and its high part summed with
// two-sum; the rounding errors, the products with the weights' low parts and
// with the differences' low parts go straight into the FP32 companion sum by
// FMA; L'xl is plain FP32 (it is 2^-24 smaller).  b and -sigma x enter the
// same accumulator, and the FP32 residual is its rounded value: r is stored in
// FP32, so only the cancellation inside the sum needs the extra precision.
//
// CYL: the y direction is periodic (rows wrap around) and its flux weight is
// one value per plane, wy[k] (the cylindrical theta direction, whose flux
// carries the radial factor of the plane).
constexpr int kResTX = 32, kResTY = 8, kResZChunk = 16;  // planes per block (at most)
constexpr int kResBX = 2 * kResTX;                       // x columns per block

// Both points of a pair run through the same operations, two FP32 values per
// instruction (f32x2: the same roundings as the scalar forms, half the issue
// slots, which bound the exact body: 209 thread instructions per point at 80%
// issue with scalar arithmetic: 124 us at 256^3, 118 us packed, when the FP32 pipe,
// which still takes a clock per value, is what is left; whole solve 546 to 537 us).
struct V2 {
  unsigned long long u;
};

__device__ __forceinline__ V2 v2(float a, float b) {
  V2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack(V2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.u));
}
__device__ __forceinline__ V2 add2(V2 a, V2 b) {
  V2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}
__device__ __forceinline__ V2 mul2(V2 a, V2 b) {
  V2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}
__device__ __forceinline__ V2 fma2(V2 a, V2 b, V2 c) {
  V2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
  return r;
}
__device__ __forceinline__ V2 minus1() { return V2{0xbf800000bf800000ull}; }
// a - b as one rounding of a + (-1) b
__device__ __forceinline__ V2 sub2(V2 a, V2 b) { return fma2(b, minus1(), a); }

struct Acc {
  V2 h, l;  // unnormalised double-float accumulators of the two points
};

// s += p, given (p exact in its high part) the low part q (or none)
template <bool LOW>
__device__ __forceinline__ void acc_add(Acc& s, V2 p, V2 q) {
  const V2 t = add2(s.h, p);
  const V2 bb = sub2(t, s.h);
  V2 e = add2(sub2(s.h, sub2(t, bb)), sub2(p, bb));
  if (LOW) e = add2(e, q);
  s.l = add2(s.l, e);
  s.h = t;
}

// a - c = d + dl exactly (Knuth two-difference)
struct Diff {
  V2 d, dl;
};

__device__ __forceinline__ Diff two_diff(V2 a, V2 c) {
  const V2 d = sub2(a, c);
  const V2 bb = sub2(d, a);
  return Diff{d, sub2(sub2(a, sub2(d, bb)), add2(c, bb))};
}

// high and low parts of a double-float weight for the two points
struct W2 {
  V2 x, y;
};

// s += w * (d + dl) for a double-float weight w: the high product enters by
// two-sum, its exact rounding error and the two small cross products by FMA
// into the low part
__device__ __forceinline__ void acc_flux(Acc& s, W2 w, Diff t) {
  const V2 p = mul2(w.x, t.d);
  const V2 e = fma2(w.x, t.d, mul2(p, minus1()));
  const V2 tt = add2(s.h, p);
  const V2 bb = sub2(tt, s.h);
  V2 l = fma2(w.x, t.dl, s.l);
  l = fma2(w.y, t.d, l);
  s.l = add2(l, add2(add2(sub2(s.h, sub2(tt, bb)), sub2(p, bb)), e));
  s.h = tt;
}

// Plain FP32 forms of the same steps, for the correction residual when the
// first residual is small (FAST): the difference rounded once, the flux
// product added by FMA to the high part, other terms added in FP32.
template <bool FAST>
__device__ __forceinline__ Diff diff_of(V2 a, V2 c) {
  if (FAST) return Diff{sub2(a, c), V2{0ull}};
  return two_diff(a, c);
}

template <bool FAST>
__device__ __forceinline__ void flux_of(Acc& s, W2 w, Diff t) {
  if (FAST)
    s.h = fma2(w.x, t.d, s.h);
  else
    acc_flux(s, w, t);
}

template <bool FAST, bool LOW>
__device__ __forceinline__ void add_of(Acc& s, V2 p, V2 q) {
  if (FAST) {
    s.h = add2(s.h, p);
    if (LOW) s.l = add2(s.l, q);
  } else {
    acc_add<LOW>(s, p, q);
  }
}

// one x pair of FP32 values (hi) and, for LO, of the low plane
struct Pair {
  V2 v, l;
};

template <bool VEC, bool LO>
__device__ __forceinline__ Pair ld_pair(const float* hi, const float* lo, int o, int d1) {
  Pair r{V2{0ull}, V2{0ull}};
  if (VEC) {
    r.v.u = *reinterpret_cast<const unsigned long long*>(hi + o);
    if (LO) r.l.u = *reinterpret_cast<const unsigned long long*>(lo + o);
  } else {
    r.v = v2(hi[o], hi[o + d1]);
    if (LO) r.l = v2(lo[o], lo[o + d1]);
  }
  return r;
}

// Two residual passes share this body.
//   MODE 0 (after the first solve):  r_1 = b - A H, with H exactly FP32; the
//     result is stored as a double-float pair (r_hi, r_lo) of FP32 planes and
//     r_hi is the next solve's input.
//   MODE 1 (after every correction): r = r_1 - A L, with L = Lh (+ Ll when LO)
//     the accumulated corrections; A is linear, so this equals b - A (H + L)
//     exactly, and only the small field L passes through the stencil.
// SIG: 0 sigma = 0, 1 sigma = 1, 2 general sigma.  MEAN: zero-flux Laplace
// problem (MODE 0 subtracts the volume-weighted mean of b; volume-weighted
// sums of the solution H (+ L) are reduced).  OUT: write the FP64 solution
// H + L.  VEC: nx even and 16-byte aligned FP64 arrays, pairs moved by vector
// accesses.
template <int MODE, int SIG, bool LO, bool MEAN, bool OUT, bool CYL, bool VEC, bool FAST>
__device__ __forceinline__ void resid_body(const ResidArgs& a, double* sh, int bx, int by, int bz, long long bid) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int i0 = 2 * (bx * kResTX + lane);
  const int j = by * kResTY + wy;
  const int k0 = bz * a.zchunk, k1 = min(nz, k0 + a.zchunk);
  const bool act0 = j < ny && i0 < nx, act1 = j < ny && i0 + 1 < nx;
  // clamped indices keep every load in bounds; a clamped neighbour is the
  // point itself (zero difference) and its flux weight is zero (a wall)
  const int ia = VEC ? min(i0, nx - 2) : min(i0, nx - 1);
  const int d1 = (VEC || ia + 1 < nx) ? 1 : 0;  // second point of the pair (scalar path)
  const int jc = min(j, ny - 1);
  const int js = jc > 0 ? jc - 1 : (CYL ? ny - 1 : 0);
  const int jn = jc + 1 < ny ? jc + 1 : (CYL ? 0 : ny - 1);
  // x of the value lane 31 needs east of its pair and lane 0 west of its pair
  const int ie = lane == kResTX - 1 ? min(i0 + 2, nx - 1) : (lane == 0 ? max(i0 - 1, 0) : ia);
  const long long oc = (long long)jc * nx + ia, os = (long long)js * nx + ia, on = (long long)jn * nx + ia;
  const long long oe = (long long)jc * nx + ie;
  const long long orr_ = (long long)jc * a.r_pitch + ia;
  float mean_h = 0.f, mean_l = 0.f;
  if (MODE == 0 && MEAN) {
    const df::F2 mb = df::from_f64(a.st->mean_b);
    mean_h = -mb.hi;
    mean_l = -mb.lo;
  }
  const int ib = ia + d1;
  auto both = [](float2 p, float2 q) { return W2{v2(p.x, q.x), v2(p.y, q.y)}; };
  const W2 wpx = both(a.wp[0][ia], a.wp[0][ib]), wmx = both(a.wm[0][ia], a.wm[0][ib]);
  W2 wpy{}, wmy{};
  float2 w0y = make_float2(0.f, 0.f);
  if (!CYL) {
    const float2 p = a.wp[1][jc], m = a.wm[1][jc];
    wpy = both(p, p);
    wmy = both(m, m);
    w0y = a.w0[1][jc];
  }
  const float2 w0xa = a.w0[0][ia], w0xb = a.w0[0][ib];
  const bool wall_xy = w0xa.x != 0.f || w0xb.x != 0.f || w0y.x != 0.f;
  df::F2 Va = df::make(0.f, 0.f), Vb = Va;
  if (MEAN) {
    const df::F2 my = ld2(a.m[1] + jc);
    Va = df::mul(ld2(a.m[0] + ia), my);
    Vb = df::mul(ld2(a.m[0] + ib), my);
  }
  __shared__ float smax[kResTY];
  float srr = 0.f, sbb = 0.f, rmax = 0.f;
  df::F2 svb = df::make(0.f, 0.f), sv = df::make(0.f, 0.f);
  // Per-row base pointers and 32-bit plane offsets (every field has fewer
  // than 2^31 elements): each access is one wide multiply-add.
  const int szi = nx * ny;           // plane stride of the [z][y][x] fields
  const int rsi = ny * a.r_pitch;    // plane stride of the residual planes
  // the field the stencil acts on: H (MODE 0) or L (MODE 1), (hi, lo) planes
  const float* uh = MODE == 0 ? a.xh : a.xl;
  const float* ul = (MODE == 1 && LO) ? a.xll : uh;
  const float* uhc = uh + oc;
  const float* uhs = uh + os;
  const float* uhn = uh + on;
  const float* uhe = uh + oe;
  const float* ulc = ul + oc;
  const float* uls = ul + os;
  const float* uln = ul + on;
  const float* ule = ul + oe;
  const double* bc = MODE == 0 ? a.b + oc : nullptr;
  const float* q1h = MODE == 1 ? a.r1 + orr_ : nullptr;
  const float* q1l = MODE == 1 ? a.r1_lo + orr_ : nullptr;
  const float* hc = (MODE == 1 && (OUT || MEAN)) ? a.xh + oc : nullptr;
  float* rc = a.r + orr_;
  float* rlc = MODE == 0 ? a.r_lo + orr_ : nullptr;
  double* outc = OUT ? a.out + oc : nullptr;
  constexpr bool LOM = MODE == 1 && LO;
  auto ldp = [&](const float* h, const float* l, int o) { return ld_pair<VEC, LOM>(h, l, o, d1); };
  auto lde = [&](int o, float& l) {
    if (LOM) l = ule[o];
    return uhe[o];
  };
  // plane k's right-hand side part: b (MODE 0, FP64) or r_1 (MODE 1, hi and lo)
  auto ldb = [&](int o, double& b0, double& b1) {
    if (VEC) {
      const double2 v = *reinterpret_cast<const double2*>(bc + o);
      b0 = v.x;
      b1 = v.y;
    } else {
      b0 = bc[o];
      b1 = bc[o + d1];
    }
  };
  auto ldr1 = [&](int o, Pair& q) { q = ld_pair<VEC, true>(q1h, q1l, o, d1); };
  auto ldh = [&](int o, float& h0, float& h1) {
    unpack(ld_pair<VEC, false>(hc, nullptr, o, d1).v, h0, h1);
  };
  // pipeline: pair C at plane k and P at k + 1, rows below (S) and above (N)
  // and the edge value E at plane k, and the right-hand side parts of plane k
  int ok = k0 * szi;                                 // plane k of the fields
  int rk = k0 * rsi;                                 // plane k of the residual planes
  Pair C = ldp(uhc, ulc, ok);
  Pair P = ldp(uhc, ulc, min(k0 + 1, nz - 1) * szi);
  Pair S = ldp(uhs, uls, ok), N = ldp(uhn, uln, ok);
  float El = 0.f;
  float E = lde(ok, El);
  double b0 = 0.0, b1 = 0.0;
  Pair Q{V2{0ull}, V2{0ull}};
  float h0 = 0.f, h1 = 0.f;
  if (MODE == 0) ldb(ok, b0, b1);
  if (MODE == 1) ldr1(rk, Q);
  if (MODE == 1 && (OUT || MEAN)) ldh(ok, h0, h1);
  // z differences across the faces below plane k (u_k - u_{k-1}; the flux takes
  // the negated weight) and the low parts of plane k-1 (LO); at k = 0 the
  // clamped plane gives zero
  Diff dz;
  V2 ml{0ull};
  {
    const Pair M = ldp(uhc, ulc, max(k0 - 1, 0) * szi);
    dz = diff_of<FAST>(C.v, M.v);
    ml = M.l;
  }
  const float2* wpz = a.wp[2];
  const float2* wmz = a.wm[2];
  const float2* w0z = a.w0[2];
  // two planes per loop pass let the register pipeline rotate without moves;
  // the exact and low-plane correction bodies keep one (their registers would
  // spill at the correction kernel's occupancy)
  constexpr int kUnroll = (MODE == 1 && (LO || !FAST)) ? 1 : 2;
#pragma unroll kUnroll
  for (int k = k0; k < k1; ++k) {
    // loads of the next plane (block-uniform guard)
    Pair P2 = P, S2 = S, N2 = N, Q2 = Q;
    float E2 = E, E2l = El;
    double b02 = 0.0, b12 = 0.0;
    float h02 = 0.f, h12 = 0.f;
    if (k + 1 < k1) {
      const int o1 = ok + szi;
      P2 = ldp(uhc, ulc, k + 2 < nz ? o1 + szi : o1);
      S2 = ldp(uhs, uls, o1);
      N2 = ldp(uhn, uln, o1);
      E2 = lde(o1, E2l);
      if (MODE == 0) ldb(o1, b02, b12);
      if (MODE == 1) ldr1(rk + rsi, Q2);
      if (MODE == 1 && (OUT || MEAN)) ldh(o1, h02, h12);
    }
    // x neighbours outside the pair: from the neighbouring lanes, or the edge value
    float ca, cb, cla = 0.f, clb = 0.f;
    unpack(C.v, ca, cb);
    const float sd = __shfl_down_sync(0xffffffffu, ca, 1);
    const float su = __shfl_up_sync(0xffffffffu, cb, 1);
    const V2 east = v2(cb, lane == kResTX - 1 ? E : sd);
    const V2 west = v2(lane == 0 ? E : su, ca);
    V2 eastl{0ull}, westl{0ull};
    if (MODE == 1 && LO) {
      unpack(C.l, cla, clb);
      const float sdl = __shfl_down_sync(0xffffffffu, cla, 1);
      const float sul = __shfl_up_sync(0xffffffffu, clb, 1);
      eastl = v2(clb, lane == kResTX - 1 ? El : sdl);
      westl = v2(lane == 0 ? El : sul, cla);
    }
    Acc A;
    df::F2 ba = df::make(0.f, 0.f), bb = ba;
    if (MODE == 0) {
      ba = df::from_f64(b0);
      bb = df::from_f64(b1);
      A = Acc{v2(ba.hi, bb.hi), v2(ba.lo, bb.lo)};
      if (MEAN) add_of<FAST, true>(A, v2(mean_h, mean_h), v2(mean_l, mean_l));
    } else {
      A = Acc{Q.v, Q.l};
    }
    if (MEAN) {
      const df::F2 mz = ld2(a.m[2] + k);
      const df::F2 Vka = df::mul(Va, mz), Vkb = df::mul(Vb, mz);
      df::F2 xa = df::make(ca, 0.f), xb = df::make(cb, 0.f);
      if (MODE == 1) {
        xa = df::two_sum(h0, ca);
        xa = df::fast_two_sum(xa.hi, xa.lo + cla);
        xb = df::two_sum(h1, cb);
        xb = df::fast_two_sum(xb.hi, xb.lo + clb);
      }
      if (act0) {
        svb = df::add(svb, df::mul(Vka, xa));
        sv = df::add(sv, Vka);
      }
      if (act1) {
        svb = df::add(svb, df::mul(Vkb, xb));
        sv = df::add(sv, Vkb);
      }
    }
    const float2 wpzk = wpz[k], wmzk = wmz[k];
    const float2 nwmz = make_float2(-wmzk.x, -wmzk.y);
    if (CYL) {
      const float2 w = a.wy[k];
      wpy = both(w, w);
      wmy = wpy;
    }
    // east, west, south, north, up, down
    flux_of<FAST>(A, wpx, diff_of<FAST>(east, C.v));
    flux_of<FAST>(A, wmx, diff_of<FAST>(west, C.v));
    flux_of<FAST>(A, wmy, diff_of<FAST>(S.v, C.v));
    flux_of<FAST>(A, wpy, diff_of<FAST>(N.v, C.v));
    const Diff du = diff_of<FAST>(P.v, C.v);
    flux_of<FAST>(A, both(wpzk, wpzk), du);
    flux_of<FAST>(A, both(nwmz, nwmz), dz);
    V2 sl{0ull};  // lambda L applied to the low parts, FP32
    if (MODE == 1 && LO) {
      sl = fma2(wpx.x, sub2(eastl, C.l), sl);
      sl = fma2(wmx.x, sub2(westl, C.l), sl);
      sl = fma2(wmy.x, sub2(S.l, C.l), sl);
      sl = fma2(wpy.x, sub2(N.l, C.l), sl);
      sl = fma2(v2(wpzk.x, wpzk.x), sub2(P.l, C.l), sl);
      sl = fma2(v2(wmzk.x, wmzk.x), sub2(ml, C.l), sl);
    }
    const float2 w0k = w0z[k];
    if (wall_xy || w0k.x != 0.f) {  // wall term: only next to a Dirichlet wall
      const df::F2 wyz = df::add(df::make(w0y.x, w0y.y), df::make(w0k.x, w0k.y));
      const df::F2 ta = df::mul(df::add(df::make(w0xa.x, w0xa.y), wyz), df::make(ca, cla));
      const df::F2 tb = df::mul(df::add(df::make(w0xb.x, w0xb.y), wyz), df::make(cb, clb));
      add_of<FAST, true>(A, v2(ta.hi, tb.hi), v2(ta.lo, tb.lo));
    }
    if (SIG == 1) {
      add_of<FAST, (MODE == 1 && LO)>(A, mul2(C.v, minus1()), mul2(C.l, minus1()));
    } else if (SIG == 2) {
      const df::F2 sg = df::make(a.sigma.x, a.sigma.y);
      const df::F2 ta = df::mul(sg, df::make(ca, cla));
      const df::F2 tb = df::mul(sg, df::make(cb, clb));
      add_of<FAST, true>(A, v2(-ta.hi, -tb.hi), v2(-ta.lo, -tb.lo));
    }
    // h + l: the rounding errors in l may exceed the cancelled h, so the pair is
    // rounded with a full two-sum
    df::F2 ra, rb;
    {
      const V2 lsum = (MODE == 1 && LO) ? add2(A.l, sl) : A.l;
      const V2 t = add2(A.h, lsum);
      unpack(t, ra.hi, rb.hi);
      ra.lo = rb.lo = 0.f;
      if (!FAST) {
        const V2 q = sub2(t, A.h);
        unpack(add2(sub2(A.h, sub2(t, q)), sub2(lsum, q)), ra.lo, rb.lo);
      }
    }
    // stores: the pair at once where both points exist
    {
      double oa = 0.0, ob = 0.0;
      if (OUT) {
        // every lane of the warp runs this (f2d_warp votes)
        oa = df::f2d_warp(h0) + (LO ? df::f2d_warp(ca) + df::f2d_warp(cla) : df::f2d_warp(ca));
        ob = df::f2d_warp(h1) + (LO ? df::f2d_warp(cb) + df::f2d_warp(clb) : df::f2d_warp(cb));
      }
      if (VEC && act0) {  // VEC: act0 implies act1
        *reinterpret_cast<float2*>(rc + rk) = make_float2(ra.hi, rb.hi);
        if (MODE == 0) *reinterpret_cast<float2*>(rlc + rk) = make_float2(ra.lo, rb.lo);
        if (OUT) *reinterpret_cast<double2*>(outc + ok) = make_double2(oa, ob);
      } else if (!VEC) {
        if (act0) {
          rc[rk] = ra.hi;
          if (MODE == 0) rlc[rk] = ra.lo;
          if (OUT) outc[ok] = oa;
        }
        if (act1) {
          rc[rk + 1] = rb.hi;
          if (MODE == 0) rlc[rk + 1] = rb.lo;
          if (OUT) outc[ok + 1] = ob;
        }
      }
    }
    if (act0) {
      srr = fmaf(ra.hi, ra.hi, srr);
      if (MODE == 0) sbb = MEAN ? fmaf(ba.hi + mean_h, ba.hi + mean_h, sbb) : fmaf(ba.hi, ba.hi, sbb);
      rmax = fmaxf(rmax, fabsf(ra.hi));
    }
    if (act1) {
      srr = fmaf(rb.hi, rb.hi, srr);
      if (MODE == 0) sbb = MEAN ? fmaf(bb.hi + mean_h, bb.hi + mean_h, sbb) : fmaf(bb.hi, bb.hi, sbb);
      rmax = fmaxf(rmax, fabsf(rb.hi));
    }
    dz = du;
    ml = C.l;
    C = P;
    P = P2;
    S = S2;
    N = N2;
    E = E2;
    El = E2l;
    b0 = b02;
    b1 = b12;
    Q = Q2;
    h0 = h02;
    h1 = h12;
    ok += szi;
    rk += rsi;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    srr += __shfl_down_sync(0xffffffffu, srr, o);
    sbb += __shfl_down_sync(0xffffffffu, sbb, o);
    rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    if (MEAN) {
      svb = df::add(svb, df::make(__shfl_down_sync(0xffffffffu, svb.hi, o), __shfl_down_sync(0xffffffffu, svb.lo, o)));
      sv = df::add(sv, df::make(__shfl_down_sync(0xffffffffu, sv.hi, o), __shfl_down_sync(0xffffffffu, sv.lo, o)));
    }
  }
  if (lane == 0) {
    sh[4 * wy + 0] = (double)srr;
    sh[4 * wy + 1] = (double)sbb;
    sh[4 * wy + 2] = MEAN ? df::to_f64(svb) : 0.0;
    sh[4 * wy + 3] = MEAN ? df::to_f64(sv) : 0.0;
    smax[wy] = rmax;
  }
  __syncthreads();
  if (wy == 0) {
    // one lane per component (a chain of FP64 adds each), one atomic per block
    if (lane < 4) {
      double t = 0.0;
      if (MEAN || lane < (MODE == 0 ? 2 : 1))
        for (int q = 0; q < kResTY; ++q) t += sh[4 * q + lane];
      a.partials[4 * bid + lane] = t;
    }
    float m = lane < kResTY ? smax[lane] : 0.f;
#pragma unroll
    for (int o = kResTY / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0 && m > 0.f) atomicMax(reinterpret_cast<unsigned int*>(a.rmax), __float_as_uint(m));
    __syncwarp();  // the record is written before thread 0 fences and takes the ticket
  }
}


// Residual grid: 64 x 8 columns per block (x pairs), `zchunk` planes marched
// per block.  Long marches amortise the loads of the planes above and below;
// grids with fewer blocks than SMs halve the march (down to 4 planes) until
// every SM has a block.  (Filling the SMs several times over made a lone
// small solve a little faster but concurrent small solves slower.)  The order
// of the reduction is fixed by the grid, which depends on the shape only.
dim3 resid_grid(int nx, int ny, int nz, int* zchunk) {
  const long long cols = (long long)((nx + kResBX - 1) / kResBX) * ((ny + kResTY - 1) / kResTY);
  int zc = kResZChunk;
  while (zc > 4 && cols * ((nz + zc - 1) / zc) < 152) zc /= 2;
  *zchunk = zc;
  return dim3((unsigned)((nx + kResBX - 1) / kResBX), (unsigned)((ny + kResTY - 1) / kResTY),
              (unsigned)((nz + zc - 1) / zc));
}

// Final reduction of the per-block partials (fixed order: deterministic) and
// the convergence bookkeeping, by one block of nt threads (t = thread index).
// kind 0: initial pass (b only): record ||b||^2 and the volume-weighted mean
// kind 1: first residual check; kind 2: later check (counts a refinement step)
__device__ void finish_block(const double* __restrict__ partials, int nblocks, DevStatus* st, double tol, int kind,
                             int want_mean, int t, int nt) {
  __shared__ double shf[4 * 32];
  double s[4] = {0, 0, 0, 0};
  // 4 half records (16 bytes) per thread in flight, fixed order; components 2
  // and 3 only where the mean is wanted
  const double2* p2 = reinterpret_cast<const double2*>(partials);
#pragma unroll 1
  for (int c = 0; c < (want_mean ? 2 : 1); ++c) {
    double x = 0.0, y = 0.0;
#pragma unroll 1
    for (int q0 = t; q0 < nblocks; q0 += 4 * nt) {
      double2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u * nt;
        v[u] = q < nblocks ? p2[2 * q + c] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (q0 - (t & 31) + u * nt < nblocks) {  // else nothing for this warp
          x += v[u].x;
          y += v[u].y;
        }
      }
    }
    if (c == 0) {
      s[0] = x;
      s[1] = y;
    } else {
      s[2] = x;
      s[3] = y;
    }
  }
  // only the warps that hold records take part
  const int w = t / 32, ln = t % 32, nw = min(nt / 32, (nblocks + 31) / 32);
  if (w < nw) {
    // lanes 0, 16, 8, 24: components 0, 1, 2, 3
    const double v = want_mean ? red::warp_sum4(s[0], s[1], s[2], s[3]) : red::warp_sum2(s[0], s[1]);
    if (ln == 0) shf[4 * w] = v;
    if (ln == 16) shf[4 * w + 1] = v;
    if (want_mean && ln == 8) shf[4 * w + 2] = v;
    if (want_mean && ln == 24) shf[4 * w + 3] = v;
  }
  __syncthreads();
  if (w != 0) return;
  // one lane per component over the warps
  double c = 0.0;
  if (ln < (want_mean ? 4 : 2))
    for (int q = 0; q < nw; ++q) c += shf[4 * q + ln];
  double tt[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) tt[q] = __shfl_sync(0xffffffffu, c, q);
  if (t != 0) return;
  if (kind == 0) {
    // the solve's status starts here (no kernel of the solve reads it before)
    st->tol_used = tol;
    st->refine_steps = 0;
    st->iters = 0;
    st->error = 0;
    st->bnorm2 = tt[1];
    if (want_mean) st->mean_b = tt[2] / tt[3];
    st->rel_res = 1.0;
    st->done = 0;
    if (!isfinite(tt[1])) {  // non-finite right-hand side: nothing more runs
      st->error = 7;
      st->done = 1;
    }
    return;
  }
  if (st->error == 7) {  // a non-finite right-hand side stays reported as such
    st->done = 1;
    return;
  }
  // the first check (r_1 = b - A H) also measures ||b||; later checks reuse it
  const double bn2 = kind == 1 ? tt[1] : st->bnorm2;
  const double rel = bn2 > 0.0 ? sqrt(tt[0] / bn2) : sqrt(tt[0]);
  if (kind == 1) {
    st->refine_steps = 0;
    st->scal[1] = rel;  // ||r_1|| / ||b||: bounds the FP32 correction residual's error
  } else {
    st->refine_steps += 1;
  }
  if (want_mean) st->scal[0] = tt[2] / tt[3];  // volume-weighted mean of the current solution
  st->rel_res = rel;
  st->bnorm2 = bn2;
  if (!isfinite(rel)) {
    st->error = 1;
    st->done = 1;
  } else {
    st->done = rel <= tol ? 1 : 0;
  }
}


}  // namespace
}  // namespace fdi
