// FP64 eigenvector transforms on the tcgen05 tensor cores.
//
// One pass of the FP64 path (Sec. 3, Eq. 25/29) applies a dense n x n matrix T
// (E_d^{-1} or E_d) to every grid line of direction d.  GB300 multiplies FP64 at
// 2 FMA/clk/SM, so on the FP64 pipe a 256^3 pass takes 6.9 ms (8.6 GFLOP at 1.25
// TFLOP/s); the same product of digits runs at the fp16 tensor rate.
//
// Method (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59, 2012: error-free
// splitting of a matrix product; on tensor cores: Mukunoki, Ozaki, Ogita,
// Imamura, ISC 2020).  Every grid line is scaled by a power of two to |x| < 1
// and rounded to a 62-bit fixed-point number, i.e. 8 signed base-256 digits (in
// [-128, 128), the leading one in [-64, 64]); the rows of T are split the same
// way at plan time.  Digits are exact in fp16, their products and the FP32 sums
// of products are integers:
//     S_L = sum_{u + v = L} sum_j T^(u)[k][j] x^(v)[j],   L = 0 .. 7,
// in units of 2^(-12 - 8 L) of the scale (the product of the powers of two above
// the line's and the row's largest entries).  For n <= 256 the bounds of
// |S_0| .. |S_4| are 2^20, 2^22, 2^23, 2^23.6 and 2^24, so these are exact for any
// input.  S_5 .. S_7 can pass 2^24 (up to 2^24.8), but only when the digits are
// near 128 and of one sign in nearly all of 256 columns (sums of random digits are
// 2^18 in root mean square); an FP32 sum then rounds by a unit, for S_5 2^-52 of the
// scale, of which the result itself is at least 2^-6.  The 36 products u + v <= 7
// leave out S_8 and beyond, 2^-58 of the scale in root mean square over 256 columns.
// The sums are added as integers and rounded to FP64 once.
//
// Accuracy is relative to the largest entry of a line, which is what the norm of a
// solution sees: on a 128-cell direction the error in a line's norm is 4-6e-17,
// that of a chain of FP64 multiply-adds 2-3e-16.  An entry 2^-k below the largest
// keeps 62 - k bits, so single results far below it are less exact than a chain's:
// the spectral coefficients of a narrow bump, half of them below 2e-16 of the
// largest, have a median relative error of 1e-3 against 1e-12.  Through the whole
// inverse the two agree point by point, since the errors of the eigenvectors weigh
// more.  Seven digits were not enough: 2e-15 on decaying lines.
//
// Layout: T is the MMA's A operand (M = 128 output modes), 64 grid lines are
// its B operand (N = 64): eight FP32 accumulators of 64 columns fill tensor
// memory, and a line is converted to digits only once per 128 modes.  Per
// 16-column step of the contraction the 36 products run from one stage of 8 digit
// planes of T (32 KB, one bulk copy from L2) and 8 of the lines (16 KB, written by
// the converters).  The digit planes of the lines follow one another, so up to
// four of them are one B operand of N = 256 rows, and its products with digit u of
// T fall into the neighbouring accumulators of levels u + v, u + v + 1, ..: 12 MMAs
// instead of 36 that each read the 4 KB of T again.
//
// Measured (GB300, x or y pass of a 256^3 field): 6.89 ms with FP64 multiply-adds,
// 0.30 ms with one MMA per product, 0.27 ms here; a whole FP64 solve of 256^3
// 28.6 -> 1.80 -> 1.70 ms, of 128^3 256 -> 248 us from the joined products.  Of the
// 34 thousand clocks of an item (64 lines, 256 columns) the MMAs take 18 (bound by
// their shared-memory reads, 120 KB per step at 128 B/clk), 11 are the epilogue,
// which holds all of tensor memory, 5 waits for operands.
//
// Warp roles of the persistent CTA (one per SM, 704 threads):
//   warp 0       bulk copies of the digit planes of T
//   warp 1       TMEM allocator and single-thread MMA issuer
//   warps 2-17   workers: read FP64 lines (cp.async, one turn ahead), split them
//                and store their digits; TMEM -> integers -> FP64 -> global store
//   warps 18-21  line exponents of the lines ahead (also pulls them into L2)
#include "fdi_internal.h"
#include "slice_transform.h"
#include "tc_common.cuh"

namespace fdi {
namespace {

constexpr int SL = 8;                         // digits
constexpr int TM = 128;                       // output modes per item (MMA M)
constexpr int TK = 16;                        // contraction columns per step (MMA K)
constexpr int STAGES = 3;
constexpr int A_SLICE = TM * TK * 2;          // 4 KB: one digit plane of T
constexpr int A_BYTES = SL * A_SLICE;
constexpr int RAW_PITCH = TK + 1;             // doubles: conflict-free row reads
constexpr int RAW_BYTES = 16 * RAW_PITCH * 8; // FP64 lines of one worker warp and step
constexpr int NWORK = 16, NEXP = 4;
constexpr int W_WORK = 2, W_EXP = W_WORK + NWORK;
constexpr int THREADS = 32 * (W_EXP + NEXP);
constexpr int EXP_BUFS = 8;                   // line tiles whose exponents are kept
constexpr int EPI_PITCH = 9;                  // doubles: 32 modes x 8 lines staging
constexpr int EPI_BYTES = 32 * EPI_PITCH * 8;
constexpr int BAR_BYTES = 512;

// shared memory for TN grid lines per item
template <int TN>
struct Smem {
  static constexpr int B_SLICE = TN * TK * 2;  // one digit plane of the lines
  static constexpr int STAGE_BYTES = A_BYTES + SL * B_SLICE;
  static constexpr int RAW_OFF = STAGES * STAGE_BYTES;
  static constexpr int EPI_OFF = RAW_OFF + NWORK * RAW_BYTES;
  static constexpr int EXP_OFF = EPI_OFF + NWORK * EPI_BYTES;
  static constexpr int BAR_OFF = EXP_OFF + EXP_BUFS * TN * 4;
  static constexpr int BYTES = BAR_OFF + BAR_BYTES;
  static_assert(BYTES + 1024 <= 232448, "shared memory budget");
  static_assert(STAGE_BYTES % 1024 == 0 && RAW_OFF % 16 == 0 && EPI_OFF % 16 == 0 && BAR_OFF % 16 == 0, "alignment");
};

struct SliceArgs {
  const double* in;
  double* out;
  const unsigned char* img;
  const int* row_exp;
  const int* skip;
  int* err;
  long long slab, rs, ks;
  unsigned R, S;
  int n, m_tiles, n_chunks, n_items, accumulate;
  long long wait_cycles;  // bound of every wait (cycles); 0: the default
};

// K-major operand with 32-byte rows in the 32-byte swizzle (8-row x 32-byte
// atoms, 256 bytes apart)
__device__ __forceinline__ uint64_t sdesc_k_sw32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(256 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;
  return d;
}

// byte offset of the 16-byte half `h` (8 fp16) of row `row`: address bit 4 ^= bit 7
__host__ __device__ __forceinline__ uint32_t sw32_offset(int row, int h) {
  return (uint32_t)(row * 32 + ((h ^ ((row >> 2) & 1)) << 4));
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ void cp_async8(uint32_t dst, const double* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// x = +-m 2^(e - 1075) on a line whose largest biased exponent is eb >= 1, as the
// fixed-point number round(x 2^(62 - (eb - 1022))), |.| < 2^62, plus 128 in every
// base-256 digit: byte q of the result is digit 7 - q plus 128.  Zeros and
// subnormal numbers have e = 1 and no leading bit.
constexpr unsigned long long kDigitBias = 0x8080808080808080ull;
__device__ __forceinline__ unsigned long long biased_digits(uint32_t lo, uint32_t hi, int eb) {
  const uint32_t f = (hi >> 20) & 0x7ffu;
  const int e = (int)max(f, 1u);
  const unsigned long long m =
      ((unsigned long long)((__funnelshift_l(lo, hi, 11) & 0x7fffffffu) | (min(f, 1u) << 31)) << 32) |
      (unsigned long long)(lo << 11);
  const int sh = eb + 1 - e;  // >= 1; one extra bit, rounded away below
  unsigned long long y;
  asm("shr.u64 %0, %1, %2;" : "=l"(y) : "l"(m), "r"((unsigned)sh));  // 0 past 63 bits
  const long long sg = (long long)((int)hi >> 31);
  const long long v = ((long long)y ^ sg) - sg;
  return (unsigned long long)((v + 1) >> 1) + kDigitBias;
}

// digit planes of two neighbouring elements as fp16 pairs: 1024 + byte by bit
// assembly, minus 1152
__device__ __forceinline__ uint32_t digit_pair(uint32_t raw) {
  __half2 h = *reinterpret_cast<__half2*>(&raw);
  const uint32_t k1152 = 0x64806480u;
  h = __hsub2(h, *reinterpret_cast<const __half2*>(&k1152));
  return *reinterpret_cast<uint32_t*>(&h);
}
template <int S>
__device__ __forceinline__ uint32_t digits_of(unsigned long long u0, unsigned long long u1) {
  const uint32_t l0 = (uint32_t)u0, l1 = (uint32_t)u1, h0 = (uint32_t)(u0 >> 32), h1 = (uint32_t)(u1 >> 32);
  // byte 7 - S of both
  constexpr int q = (SL - 1 - S) & 3;
  constexpr unsigned sel = 0x5410u + 0x1111u * q;  // bytes q, q + 1 of each word (the upper one is masked)
  const uint32_t w = __byte_perm(S < 4 ? h0 : l0, S < 4 ? h1 : l1, q == 3 ? 0x7733u : sel);
  return digit_pair((w & 0x00ff00ffu) | 0x64006400u);
}

// the eight level sums (integers held in FP32; level L weighs 2^(8 (14 - L)) in
// units of the two fixed-point numbers) as one 64-bit integer of 61 or more
// significant bits, rounded to FP64; be0: biased exponent of 2^63 in units of
// 2^88.  Results outside the normal range are left to the caller (`off`): no
// branch, so the outputs of a thread interleave.
__device__ __forceinline__ double levels_to_f64(const float (&s)[SL], int be0, bool& off) {
  // |s_0|, |s_1| <= 2^22: integers by a magic addition
  const int f0 = __float_as_int(s[0] + 12582912.f), f1 = __float_as_int(s[1] + 12582912.f);
  const int a = (f0 << 8) + (f1 - (int)(0x4b400000u * 257u));
  const int i2 = __float2int_rn(s[2]), i3 = __float2int_rn(s[3]), i4 = __float2int_rn(s[4]), i5 = __float2int_rn(s[5]);
  const int i6 = __float2int_rn(fmaf(s[7], 0.00390625f, s[6]));
  // levels 0-3 in units of 2^88 (|.| <= 2^44.1), levels 4-7 in units of 2^64 (<= 2^40.1)
  const long long t = (long long)a * 65536 + ((long long)i2 * 256 + i3);
  const long long w = (long long)i4 * 65536 + ((long long)i5 * 256 + i6);
  // left-justify the upper part (at most by the 24 bits between the units)
  const long long st = t >> 63;
  const int j = min(24, __clzll((t ^ st) - st) - 2);
  const long long x = (t << j) + (w >> (24 - j));
  const long long sx = x >> 63;
  unsigned long long m = (unsigned long long)((x ^ sx) - sx);
  const int lz = __clzll((long long)m);
  m <<= lz & 63;
  const int be = be0 - j - lz;
  const unsigned long long q = m >> 11;
  const unsigned up = (((unsigned)m & 0x7ffu) + ((unsigned)q & 1u) > 0x400u) ? 1u : 0u;  // nearest, ties to even
  const unsigned long long bits =
      ((unsigned long long)(unsigned)(be - 1) << 52) + q + up + ((unsigned long long)sx & 0x8000000000000000ull);
  off |= x != 0 && (unsigned)(be - 1) > 2045u;
  return x != 0 ? __longlong_as_double((long long)bits) : 0.0;
}

// the same for results that overflow or underflow FP64's normal range
__device__ __noinline__ double levels_to_f64_slow(const float* s, int be0) {
  double v = 0.0;
  for (int l = SL - 1; l >= 0; --l) v += scalbn((double)s[l], 24 - 8 * l);  // in units of 2^88
  return scalbn(v, be0 - 1086);
}

template <int TN>
__global__ void __launch_bounds__(THREADS, 1) k_slice_transform(const SliceArgs a) {
  using SM = Smem<TN>;
  constexpr int WPG = TN / 16;        // worker warps that convert one step together
  constexpr int GROUPS = NWORK / WPG;
  constexpr int CW = TN / 4;          // lines per worker in the epilogue
  extern __shared__ __align__(1024) uint8_t smem[];
  // a correction round that may be idle asks first: the idle launch then costs
  // neither barriers nor TMEM (FP64 Stokes, 48 x 64 x 40: 3.72 -> 3.64 ms).  A first round has no flag and sets
  // itself up while the kernel before it drains.
  if (a.skip) {
    pdl_wait();
    if (*a.skip) return;
  }
  if ((tc::smem_u32(smem) & 1023u) != 0u) {  // the swizzled stages need the alignment
    pdl_wait();
    if (threadIdx.x == 0) atomicExch(a.err, 7);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::BAR_OFF);
  uint64_t* full = bars;                       // digit planes of T landed (bulk-copy bytes)
  uint64_t* conv = full + STAGES;              // digit planes of the lines written (WPG warps)
  // stage free again (one commit of the MMAs that read it): one barrier per
  // group of workers, not per stage, since a group must see every phase of a
  // barrier it waits on (a parity wait that skips phases can pass too early).
  // Step g >= STAGES waits for barrier g % GROUPS, committed by step g - STAGES.
  uint64_t* freed = conv + STAGES;
  uint64_t* accf = freed + GROUPS;             // accumulators complete
  uint64_t* acce = accf + 1;                   // accumulators drained (NWORK warps)
  uint64_t* expf_ = accf + 2;                  // line exponents written (NEXP warps)
  uint64_t* expe = expf_ + EXP_BUFS;           // line exponents no longer needed (NWORK warps)
  uint64_t* mma_drain = expe + EXP_BUFS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_drain + 1);
  static_assert((2 * STAGES + GROUPS + 2 + 2 * EXP_BUFS + 2) * 8 <= BAR_BYTES, "barriers");
  static_assert(GROUPS >= STAGES, "a freed barrier completes at most once per step of its group");
  int* s_exp = reinterpret_cast<int*>(smem + SM::EXP_OFF);  // [EXP_BUFS][TN]
  __shared__ volatile int s_abort;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const long long wl = a.wait_cycles > 0 ? a.wait_cycles : tc::kWaitCycles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&conv[s], WPG);
    }
    for (int b = 0; b < GROUPS; ++b) tc::mbar_init(&freed[b], 1);
    tc::mbar_init(accf, 1);
    tc::mbar_init(acce, NWORK);
    for (int b = 0; b < EXP_BUFS; ++b) {
      tc::mbar_init(&expf_[b], NEXP);
      tc::mbar_init(&expe[b], NWORK);
    }
    tc::mbar_init(mma_drain, 1);
    s_abort = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(tmem_slot, 8 * TN);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // nothing above touches data of the kernel before this one in the stream
  pdl_wait();

  // items (line tile, mode tile), mode tile fastest; a CTA takes a contiguous run
  const int i0 = (int)((long long)blockIdx.x * a.n_items / gridDim.x);
  const int i1 = (int)((long long)(blockIdx.x + 1) * a.n_items / gridDim.x);
  const int items = i1 - i0, nK = a.n_chunks;
  const int lt0 = i0 / a.m_tiles;
  const bool kmajor = a.ks == 1;  // lines contiguous (x), else neighbouring lines are
  // waits until the stage of step g may be written
  auto stage_free = [&](int g) -> bool {
    if (g < STAGES) return true;
    const int b = g % GROUPS, phase = g / GROUPS - (b < STAGES ? 1 : 0);
    return tc::mbar_wait(&freed[b], (uint32_t)(phase & 1), &s_abort, wl);
  };

  if (warp == 0) {
    if (tc::elect_one()) {
      uint32_t g = 0;
      for (int it = 0; it < items && !s_abort; ++it) {
        const int mt = (i0 + it) % a.m_tiles;
        const unsigned char* src = a.img + (size_t)mt * nK * A_BYTES;
        for (int kc = 0; kc < nK; ++kc, ++g) {
          const int s = g % STAGES;
          if (!stage_free((int)g)) {
            atomicExch(a.err, 1);
            break;
          }
          tc::mbar_expect_tx(&full[s], A_BYTES);
          tc::bulk_load(tc::smem_u32(smem + s * SM::STAGE_BYTES), src + (size_t)kc * A_BYTES, A_BYTES, &full[s]);
        }
      }
      // copies issued last may still be writing shared memory after a failure
      for (uint32_t g2 = g > STAGES ? g - STAGES : 0; g2 < g; ++g2)
        tc::mbar_drain(&full[g2 % STAGES], (g2 / STAGES) & 1);
    }
  } else if (warp == 1) {
    // one elected thread (under a lane test 56-76 clocks per N = 64 MMA instead of 35)
    if (tc::elect_one()) {
      constexpr int NPL = 256 / TN;  // digit planes of the lines per MMA (N <= 256)
      const uint32_t s_base = tc::smem_u32(smem);
      uint32_t g = 0;
      for (int it = 0; it < items && !s_abort; ++it) {
        if (!tc::mbar_wait(acce, (uint32_t)(it & 1) ^ 1u, &s_abort, wl)) {
          atomicExch(a.err, 2);
          break;
        }
        tc::tc_fence_after();
        bool ok = true;
        for (int kc = 0; kc < nK; ++kc, ++g) {
          const int s = g % STAGES;
          const uint32_t ph = (g / STAGES) & 1;
          if (!tc::mbar_wait(&full[s], ph, &s_abort, wl) || !tc::mbar_wait(&conv[s], ph, &s_abort, wl)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t sa = s_base + s * SM::STAGE_BYTES, sb = sa + A_BYTES;
          // digit u of T times digit v of the lines goes to level u + v; the
          // first step's u = 0 products start every level.  Up to 256 rows of
          // the digit planes v, v + 1, .. are one B operand, whose products with
          // digit u land in the neighbouring columns of levels u + v, u + v + 1, ..
#pragma unroll
          for (int u = 0; u < SL; ++u) {
            const uint64_t da = sdesc_k_sw32(sa + u * A_SLICE);
            const uint32_t acc = (kc > 0 || u > 0) ? 1u : 0u;
#pragma unroll
            for (int v = 0; v < SL - u; v += NPL) {
              const int planes = SL - u - v < NPL ? SL - u - v : NPL;
              const uint32_t d = tmem + (uint32_t)((u + v) * TN);
              const uint64_t db = sdesc_k_sw32(sb + v * SM::B_SLICE);
              tc::mma_f16(d, da, db, tc::idesc_f16_f32(TM, planes * TN), acc);
            }
          }
          tc::mma_commit(&freed[(g + STAGES) % GROUPS]);
        }
        if (!ok) {
          s_abort = 1;
          atomicExch(a.err, 3);
          break;
        }
        tc::mma_commit(accf);
      }
      tc::mma_commit(mma_drain);
      tc::mbar_drain(mma_drain, 0);
    }
  } else if (warp < W_EXP) {
    // ---------------- workers: converters and epilogue ----------------
    // WPG warps convert one step together, 16 lines x 16 columns each; the
    // groups take turns.  The FP64 values of a warp's next step are loaded
    // while the other groups convert.  An item's epilogue comes after the
    // conversion of the first STAGES steps of the next item, so the MMAs resume
    // as soon as the accumulators are free.
    const int ww = warp - W_WORK, grp = ww / WPG, wg = ww % WPG;
    uint8_t* raw = smem + SM::RAW_OFF + ww * RAW_BYTES;
    const uint32_t raw_dst = tc::smem_u32(raw);
    const int total = items * nK;
    const int line = lane & 15, half = lane >> 4;
    // load position
    int l_it = grp / nK, l_kc = grp % nK, l_lt = -1;
    const double* l_base = a.in;
    bool l_ok = false;
    auto issue = [&](int gi) {
      if (gi < total) {
        const int lt = (i0 + l_it) / a.m_tiles;
        const unsigned r0 = (unsigned)lt * TN + 16u * wg;
        const int k0 = l_kc * TK;
        if (kmajor) {
          // half-warps read 16 columns (128 bytes) of a line each
          const int k = k0 + line;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int ln = 2 * q + half;
            const bool ok = r0 + ln < a.R && k < a.n;
            cp_async8(raw_dst + (ln * RAW_PITCH + line) * 8, ok ? a.in + (long long)(r0 + ln) * a.rs + k : a.in, ok);
          }
        } else {
          // 16 neighbouring lines of one column per half-warp
          if (lt != l_lt) {
            const unsigned r = r0 + line;
            l_ok = r < a.R;
            l_base = l_ok ? a.in + (long long)(r / a.S) * a.slab + (long long)(r % a.S) * a.rs : a.in;
            l_lt = lt;
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int k = 2 * q + half;
            const bool ok = l_ok && k0 + k < a.n;
            cp_async8(raw_dst + (line * RAW_PITCH + k) * 8, ok ? l_base + (long long)(k0 + k) * a.ks : a.in, ok);
          }
        }
        l_kc += GROUPS;
        while (l_kc >= nK) {
          l_kc -= nK;
          ++l_it;
        }
      }
      cp_async_commit();
    };
    const int tq = warp & 3, cg = ww >> 2;  // tensor-memory quarter (32 modes), group of CW lines
    double* tp = reinterpret_cast<double*>(smem + SM::EPI_OFF + ww * EPI_BYTES);
    auto epilogue = [&](int it) -> bool {
      const int lt = (i0 + it) / a.m_tiles, mt = (i0 + it) % a.m_tiles, ltq = lt - lt0, eb_buf = ltq % EXP_BUFS;
      if (!tc::together(tc::mbar_wait(&expf_[eb_buf], (ltq / EXP_BUFS) & 1, &s_abort, wl) &&
                        tc::mbar_wait(accf, (uint32_t)(it & 1), &s_abort, wl))) {
        atomicExch(a.err, 5);
        return false;
      }
      tc::tc_fence_after();
      const int* eb = s_exp + eb_buf * TN + CW * cg;
      const int k0 = mt * TM + 32 * tq, k = k0 + lane;
      const unsigned r0 = (unsigned)lt * TN + (unsigned)(CW * cg);
      if (k0 < a.n && r0 < a.R) {
        const int ek = k < a.n ? a.row_exp[k] - 994 : 0;
#pragma unroll 1
        for (int c0 = 0; c0 < CW; c0 += 8) {
          if (!kmajor) __syncwarp();
#pragma unroll 1
          for (int c1 = 0; c1 < 8; c1 += 4) {
            float v[SL][4];
#pragma unroll
            for (int l = 0; l < SL; ++l)
              tmem_ld4(tmem + ((uint32_t)(32 * tq) << 16) + (uint32_t)(l * TN + CW * cg + c0 + c1), v[l]);
            tc::tmem_ld_wait();
            double o[4];
            bool off = false;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float s[SL] = {v[0][c], v[1][c], v[2][c], v[3][c], v[4][c], v[5][c], v[6][c], v[7][c]};
              o[c] = levels_to_f64(s, eb[c0 + c1 + c] + ek, off);
            }
            if (off) {
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const float s[SL] = {v[0][c], v[1][c], v[2][c], v[3][c], v[4][c], v[5][c], v[6][c], v[7][c]};
                o[c] = levels_to_f64_slow(s, eb[c0 + c1 + c] + ek);
              }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)  // a non-finite entry in the line
              if (eb[c0 + c1 + c] == 0x7ff) o[c] = __longlong_as_double(0x7ff8000000000000ll);
            if (kmajor) {
              // 32 modes of one line are contiguous
              if (k < a.n) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const unsigned r = r0 + c0 + c1 + c;
                  if (r < a.R) {
                    double* dst = a.out + (long long)r * a.rs + k;
                    *dst = a.accumulate ? *dst + o[c] : o[c];
                  }
                }
              }
            } else {
#pragma unroll
              for (int c = 0; c < 4; ++c) tp[lane * EPI_PITCH + c1 + c] = o[c];
            }
          }
          if (!kmajor) {
            // through shared memory: 8 neighbouring lines of 4 modes per store
            __syncwarp();
            const int cl = lane & 7;
            const unsigned r = r0 + c0 + cl;
            if (r < a.R) {
              double* base = a.out + (long long)(r / a.S) * a.slab + (long long)(r % a.S) * a.rs;
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const int kl = 4 * j + (lane >> 3);
                if (k0 + kl < a.n) {
                  double* dst = base + (long long)(k0 + kl) * a.ks;
                  const double w = tp[kl * EPI_PITCH + cl];
                  *dst = a.accumulate ? *dst + w : w;
                }
              }
            }
          }
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        tc::mbar_arrive(acce);
        if (mt == a.m_tiles - 1 || it == items - 1) tc::mbar_arrive(&expe[eb_buf]);
      }
      return true;
    };

    issue(grp);
    int it = grp / nK, kc = grp % nK, ltq = -1, eb = 0, done = 0;
    bool ok = true;
    for (int gi = grp; gi < total; gi += GROUPS) {
      while (done < items && gi >= (done + 1) * nK + STAGES && ok) ok = epilogue(done++);
      if (!ok) break;
      const int s = gi % STAGES;
      cp_async_wait<0>();
      __syncwarp();
      uint2 x[8];
      const uint2* src = reinterpret_cast<const uint2*>(raw) + line * RAW_PITCH + half * 8;
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = src[q];
      __syncwarp();
      issue(gi + GROUPS);
      const int want = (i0 + it) / a.m_tiles - lt0;
      if (want != ltq) {
        ltq = want;
        ok = tc::together(tc::mbar_wait(&expf_[ltq % EXP_BUFS], (ltq / EXP_BUFS) & 1, &s_abort, wl));
        eb = s_exp[(ltq % EXP_BUFS) * TN + 16 * wg + line];
      }
      unsigned long long u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = biased_digits(x[q].x, x[q].y, eb);
      if (!ok || !tc::together(stage_free(gi))) {
        atomicExch(a.err, 4);
        break;
      }
      uint8_t* st = smem + s * SM::STAGE_BYTES + A_BYTES + sw32_offset(16 * wg + line, half);
#define FDI_STORE_DIGITS(S)                                                                   \
  *reinterpret_cast<uint4*>(st + S * SM::B_SLICE) =                                           \
      make_uint4(digits_of<S>(u[0], u[1]), digits_of<S>(u[2], u[3]), digits_of<S>(u[4], u[5]), \
                 digits_of<S>(u[6], u[7]))
      FDI_STORE_DIGITS(0);
      FDI_STORE_DIGITS(1);
      FDI_STORE_DIGITS(2);
      FDI_STORE_DIGITS(3);
      FDI_STORE_DIGITS(4);
      FDI_STORE_DIGITS(5);
      FDI_STORE_DIGITS(6);
      FDI_STORE_DIGITS(7);
#undef FDI_STORE_DIGITS
      tc::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&conv[s]);
      kc += GROUPS;
      while (kc >= nK) {
        kc -= nK;
        ++it;
      }
    }
    while (done < items && ok) ok = epilogue(done++);
    cp_async_wait<0>();
  } else {
    // ---------------- line exponents ----------------
    // biased exponent of the largest |x| of every line (its high words), up to
    // EXP_BUFS line tiles ahead; also brings the lines into L2
    constexpr int LPW = TN / NEXP;  // lines per warp
    const int w = warp - W_EXP;
    const int last = items > 0 ? (i0 + items - 1) / a.m_tiles - lt0 : -1;
    const uint32_t* hi = reinterpret_cast<const uint32_t*>(a.in) + 1;
    for (int ltq = 0; ltq <= last; ++ltq) {
      const int b = ltq % EXP_BUFS;
      if (!tc::together(tc::mbar_wait(&expe[b], ((ltq / EXP_BUFS) & 1) ^ 1, &s_abort, wl))) {
        atomicExch(a.err, 6);
        break;
      }
      const unsigned r0 = (unsigned)(lt0 + ltq) * TN + (unsigned)(LPW * w);
      if (kmajor) {
#pragma unroll 1
        for (int l0 = 0; l0 < LPW; l0 += 8) {
          uint32_t mx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
          for (int k = lane; k < a.n; k += 32)
#pragma unroll
            for (int l = 0; l < 8; ++l) {
              const unsigned r = r0 + l0 + l;
              if (r < a.R) mx[l] = max(mx[l], hi[2 * ((long long)r * a.rs + k)] & 0x7fffffffu);
            }
#pragma unroll
          for (int l = 0; l < 8; ++l) {
            const uint32_t m = __reduce_max_sync(0xffffffffu, mx[l]);
            if (lane == 0) s_exp[b * TN + LPW * w + l0 + l] = max((int)(m >> 20), 1);
          }
        }
      } else {
        const int line = lane % LPW;
        const unsigned r = r0 + line;
        uint32_t mx = 0;
        if (r < a.R) {
          const uint32_t* p = hi + 2 * ((long long)(r / a.S) * a.slab + (long long)(r % a.S) * a.rs);
#pragma unroll 16
          for (int k = lane / LPW; k < a.n; k += 32 / LPW) mx = max(mx, p[2 * (long long)k * a.ks] & 0x7fffffffu);
        }
#pragma unroll
        for (int o = LPW; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane < LPW) s_exp[b * TN + LPW * w + line] = max((int)(mx >> 20), 1);
      }
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&expf_[b]);
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 8 * TN);
  }
}

// digit planes of a matrix row (one block per row of the padded tiles)
__global__ void k_slice_matrix(const double* __restrict__ T, int n, int n_chunks, unsigned char* __restrict__ img,
                               int* __restrict__ row_exp) {
  const int k = blockIdx.x;
  __shared__ unsigned s_max;
  if (threadIdx.x == 0) s_max = 0;
  __syncthreads();
  unsigned mx = 0;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    if (k < n) mx = max(mx, (unsigned)__double2hiint(T[(size_t)k * n + j]) & 0x7fffffffu);
  atomicMax(&s_max, mx);
  __syncthreads();
  const int eb = max((int)(s_max >> 20), 1);
  if (threadIdx.x == 0) row_exp[k] = eb;
  for (int j = threadIdx.x; j < n_chunks * TK; j += blockDim.x) {
    const double t = (k < n && j < n) ? T[(size_t)k * n + j] : 0.0;
    const unsigned long long u = biased_digits((uint32_t)__double2loint(t), (uint32_t)__double2hiint(t), eb);
    unsigned char* base = img + ((size_t)(k / TM) * n_chunks + j / TK) * A_BYTES +
                          sw32_offset(k % TM, (j % TK) >> 3) + (j & 7) * 2;
    for (int d = 0; d < SL; ++d) {
      const int byte = (int)((u >> (8 * (SL - 1 - d))) & 0xff);
      *reinterpret_cast<__half*>(base + (size_t)d * A_SLICE) = __int2half_rn(byte - 128);
    }
  }
}

#define FDI_TRY(expr)            \
  do {                           \
    fdi_status _s = (expr);      \
    if (_s != FDI_OK) return _s; \
  } while (0)

fdi_status prepare_matrix(fdi_plan* p, const double* T, int n, SliceMatrix* m, cudaStream_t s) {
  m->n = n;
  m->m_tiles = (n + TM - 1) / TM;
  m->n_chunks = (n + TK - 1) / TK;
  cudaError_t e = cudaMalloc(&m->img, (size_t)m->m_tiles * m->n_chunks * A_BYTES);
  if (e == cudaSuccess) e = cudaMalloc(&m->row_exp, (size_t)m->m_tiles * TM * sizeof(int));
  if (e != cudaSuccess) {
    cudaGetLastError();  // reported here, not by the next launch check
    set_error(std::string("digit planes of a transform: ") + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? FDI_ERR_OUT_OF_MEMORY : FDI_ERR_CUDA;
  }
  k_slice_matrix<<<m->m_tiles * TM, 256, 0, s>>>(T, n, m->n_chunks, m->img, m->row_exp);
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

}  // namespace

fdi_status slice_prepare_axis(fdi_plan* p, Axis* ax, cudaStream_t s) {
  if (ax->slices) return FDI_OK;
  FDI_CUDA_TRY(cudaFuncSetAttribute(k_slice_transform<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<64>::BYTES));
  FDI_CUDA_TRY(cudaFuncSetAttribute(k_slice_transform<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<32>::BYTES));
  SliceAxis* sa = new SliceAxis();
  ax->slices = sa;
  FDI_TRY(prepare_matrix(p, ax->Einv, ax->n, &sa->fwd, s));
  return prepare_matrix(p, ax->E, ax->n, &sa->bwd, s);
}

void slice_free_axis(Axis* ax) {
  SliceAxis* sa = static_cast<SliceAxis*>(ax->slices);
  if (!sa) return;
  for (SliceMatrix* m : {&sa->fwd, &sa->bwd}) {
    if (m->img) cudaFree(m->img);
    if (m->row_exp) cudaFree(m->row_exp);
  }
  delete sa;
  ax->slices = nullptr;
}

fdi_status launch_slice_transform(fdi_plan* p, const SliceMatrix& m, const double* in, double* out,
                                  const SliceLines& g, bool accumulate, bool pdl, const int* skip,
                                  cudaStream_t s) {
  SliceArgs a{};
  a.in = in;
  a.out = out;
  a.img = m.img;
  a.row_exp = m.row_exp;
  a.skip = skip;
  a.err = p->d_err;
  a.slab = g.slab;
  a.rs = g.rs;
  a.ks = g.ks;
  a.R = (unsigned)g.R;
  a.S = (unsigned)g.S;
  a.n = m.n;
  a.m_tiles = m.m_tiles;
  a.n_chunks = m.n_chunks;
  a.accumulate = accumulate ? 1 : 0;
  a.wait_cycles = p->wait_cycles;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
  // 64 lines per item, or 32 where that leaves SMs without work
  const bool wide = (g.R + 63) / 64 * m.m_tiles >= sms;
  const int tn = wide ? 64 : 32;
  a.n_items = (int)((g.R + tn - 1) / tn) * m.m_tiles;
  const int grid = a.n_items < sms ? a.n_items : sms;
  FDI_CUDA_TRY(launch_pdl(pdl && p->pdl, wide ? k_slice_transform<64> : k_slice_transform<32>, dim3((unsigned)grid),
                          dim3(THREADS), (size_t)(wide ? Smem<64>::BYTES : Smem<32>::BYTES), s, a));
  FDI_LAUNCH_CHECK(p);
  return FDI_OK;
}

}  // namespace fdi
