// Tall-skinny products of the BMG cycle on the 5th-generation tensor cores (tcgen05),
// with float64-class accuracy from exact BF16 digit slices.
//
//   Gram      G = X^T Y        X, Y: [n][ld] blocks, contraction over the n rows
//             (the Rayleigh-Ritz block matrices X^T A X, X^T M X of Sec. 4.1)
//   expand    U = Z + X Yx     X: [n][ld], Yx: k x k, contraction over k
//             (Ritz vectors in V_{h1} + span X: U = Q Y_c + X Y_x)
//
// GB300 retires float64 at about 1/64 of its float32 rate, while its tensor cores
// multiply BF16 at petaflop rates.  Both products are therefore formed from integer
// digits, in the manner of Ozaki, Ogita, Oishi & Rump (2012, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication"), but with the exactness carried by integer arithmetic:
//
//  1. Scaling.  Every value x of a scaling group (Gram: one column of X or Y over a
//     window of 256 rows; expand: one row of X over its k values, one column of Yx)
//     with group exponent E (the largest biased exponent in the group, so that
//     |x| < 2^(E - bias + 1)) is turned into the integer V = round(x 2^(F - E + bias
//     - 1)), |V| <= 2^F, F = 7 S - 1.
//  2. Digits.  V = sum_{s=1..S} d_s 2^(7 (S - s)) with balanced digits d_s in [-64, 64],
//     each stored with its weight as a BF16 value exactly (struct Digits).
//  3. Products.  For every digit pair (s, t) with s + t <= T the tensor cores
//     accumulate sum_r d_s(x_r) d_t(y_r) in float32 in tensor memory; pairs with
//     the same diagonal s + t share an accumulator and a scale.  A diagonal holds at most
//     8 pairs over at most 256 terms of magnitude <= 2^12, so every partial sum is a
//     power of two times an integer of magnitude <= 2^23 and the float32 accumulation is
//     exact.
//  4. Combination.  The diagonals of a window are read back (tcgen05.ld), turned
//     into int32 exactly, and combined with shifts into one 96-bit integer per output
//     element; windows are added after aligning their exponents.  Only the last step, the
//     conversion to float64, rounds.
//
// Error: dropping the pairs s + t > T and rounding V leave an error below about
// (T - 1) 2^(-7 (T - 1)) K max|x| max|y| per window of K terms: 2^-53 for float64
// blocks (S = 8, T = 9, 36 pairs), 2^-33 for float32 blocks (S = 5, T = 6,
// 15 pairs), where the data themselves carry 2^-24.
//
// Kernel structure (one CTA per SM: 192 KB of shared memory, up to 512 TMEM
// columns).  Operand digits are written by 16 worker warps into shared memory in the
// no-swizzle K-major core-matrix layout (8 rows x 16 bytes per core matrix), two
// stages; one thread of a seventeenth warp issues tcgen05.mma (kind::f16, BF16 x BF16 ->
// FP32, M = 128, N = 128 to 256) and commits to an mbarrier per stage, so that the digits of
// the next 32-row sub-chunk are formed while the tensor cores work on the current one;
// three more warps gather the exponents ahead.  Every wait is bounded (about 2 s of clock);
// on expiry the kernel raises *err, waits a bounded time more, frees its tensor memory and
// returns.
//
// Measured, 655362 x 128, float64 (float32): Gram 1720 -> 1030 us (1200 -> 578),
// expansion 2130 -> 1430 us (1270 -> 705).  The largest parts of it: one wide MMA for several
// digit planes of B, exponents by their own warps from L2 with 16-byte loads, digits by float32
// additions.  One base and N for all MMAs of a group of accumulators (issue_mmas) adds a third
// of zero products: 1002 and 1387 us (533 and 665) without it.  What bounds the float64 forms
// now: the readback's and the digits' integer work at four warps a scheduler (before that
// change, the Gram took 950 us without the MMAs and 980 us without the readback).
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace bmg {
namespace {

constexpr int kWorkers = 512;             // 16 warps forming digits and reading TMEM back; warps w,
                                         // w+4, w+8, w+12 share TMEM lanes
constexpr int kMmaWarp = kWorkers / 32;  // one warp that issues the MMAs
constexpr int kScanWarps = 3;            // and three that gather the exponents ahead (registers are
                                         // allocated for 20 warps as for 17)
constexpr int kScan0 = kMmaWarp + 1;
constexpr int kTcThreads = kWorkers + 32 + 32 * kScanWarps;
constexpr int kKsub = 32;                // K rows per sub-chunk (two MMA K-steps of 16)
constexpr int kWindow = 256;             // K rows per exact accumulation window (Gram)
constexpr int kNB = 64;                  // output columns per CTA (N of the MMA)
constexpr int kBeta = 7;                 // digit width
constexpr long long kWaitCycles = 4000000000LL;   // ~2 s at 2 GHz

// Digit layout of one operand (rows x kKsub, BF16, K-major, no swizzle).
constexpr int kAPlane = 128 * kKsub * 2;  // bytes per digit plane of the 128-row operand
constexpr int kBPlane = kNB * kKsub * 2;  // bytes per digit plane of the 64-row operand
static_assert(kBPlane == (kNB / 8) * kKsub * 16, "planes of B one 8-row stride apart (issue_mmas)");

// Planes of the 64-row operand that one MMA multiplies (its N is kNB times that), and the zero
// planes in front of them (issue_mmas); S digits: 8 of float64 blocks, 5 of float32 blocks.
__host__ __device__ constexpr int mma_planes(int S) { return S == 8 ? 4 : 3; }
__host__ __device__ constexpr int zero_planes(int S) { return mma_planes(S) - 1; }
__host__ __device__ constexpr int stage_bytes(int S) { return S * kAPlane + (zero_planes(S) + S) * kBPlane; }
// offset of the first digit plane of the 64-row operand in a stage
__host__ __device__ constexpr int b_offset(int S) { return S * kAPlane + zero_planes(S) * kBPlane; }

// byte offset of the 8-element K-group starting at (row, k0) (k0 % 8 == 0)
__device__ __forceinline__ int cm_off(int row, int k0) {
  return (row >> 3) * (kKsub * 16) + (k0 >> 3) * 128 + (row & 7) * 16;
}

// ------------------------------------------------------------ PTX wrappers ----
__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (tcgen05): start address, leading byte offset
// (distance of the two K-adjacent core matrices), stride byte offset (distance of
// 8-row groups), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// Instruction descriptor, kind::f16: BF16 A and B (K-major), FP32 D, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Waits for the completion of the phase with the given parity; false after `limit`
// clocks without it (kWaitCycles, about 2 s, except in the timeout self-tests).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// int32 of a float32 holding an integer (exact: |value| <= 2^23 here)
__device__ __forceinline__ int f2i_exact(uint32_t bits) { return __float2int_rn(__uint_as_float(bits)); }

// ------------------------------------------------------------ digits ----------
template <typename T> struct Fmt;
// emax: the biased exponent of Inf and NaN.  A group holding one has that group
// exponent, and every output it contributes to is NaN.
template <> struct Fmt<double> {
  static constexpr int bias = 1023, emax = 2047;
  // the words of 2 (float32: 4) columns of a row that hold the exponents, `cols` of them
  // valid (vec: the others are read too, and the caller masks them)
  __device__ static void words(const double* p, int cols, bool vec, uint32_t (&w)[2]) {
    if (vec) {             // the 16 bytes lie inside the row: its stride is a multiple of 16
      const uint4 t = *reinterpret_cast<const uint4*>(p);
      w[0] = t.y;
      w[1] = t.w;
    } else {
      w[0] = word(p);
      w[1] = cols >= 2 ? word(p + 1) : 0u;
    }
  }
  __device__ static int expo(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
  // the word of *p that holds the exponent, and the exponent in it
  __device__ static uint32_t word(const double* p) { return reinterpret_cast<const uint32_t*>(p)[1]; }
  __device__ static int expo_of(uint32_t w) { return (int)((w >> 20) & 0x7FF); }
};
template <> struct Fmt<float> {
  static constexpr int bias = 127, emax = 255;
  __device__ static void words(const float* p, int cols, bool vec, uint32_t (&w)[4]) {
    if (vec) {
      const uint4 t = *reinterpret_cast<const uint4*>(p);
      w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) w[q] = q < cols ? word(p + q) : 0u;
    }
  }
  __device__ static int expo(float x) { return (int)((__float_as_uint(x) >> 23) & 0xFF); }
  __device__ static uint32_t word(const float* p) { return *reinterpret_cast<const uint32_t*>(p); }
  __device__ static int expo_of(uint32_t w) { return (int)((w >> 23) & 0xFF); }
};

// two float32 values of at most 8 significant bits as one BF16 pair (exact): the top
// halves of their bit patterns, the first in the low half
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
__host__ __device__ constexpr float pow2f(int e) {
  float v = 1.f;
  for (int q = 0; q < (e < 0 ? -e : e); ++q) v = e < 0 ? v * 0.5f : v * 2.f;
  return v;
}
// x rounded to a multiple of 2^e (|x| < 2^(e + 22)), and the remainder left in x
template <int E>
__device__ __forceinline__ float take_digit(float& x) {
  constexpr float M = 1.5f * pow2f(23 + E);
  const float d = __fsub_rn(__fadd_rn(x, M), M);
  x = __fsub_rn(x, d);
  return d;
}
// one plane of 8 digits (16 bytes)
__device__ __forceinline__ void store_plane(unsigned char* dst, const float (&d)[8]) {
  *reinterpret_cast<uint4*>(dst) = make_uint4(pack_bf16(d[0], d[1]), pack_bf16(d[2], d[3]), pack_bf16(d[4], d[5]),
                                              pack_bf16(d[6], d[7]));
}
template <int E>
__device__ __forceinline__ void take_plane(float (&x)[8], unsigned char* dst) {
  float d[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) d[q] = take_digit<E>(x[q]);
  store_plane(dst, d);
}

// Digits of 8 values of one scaling group (exponent E): plane s (s = 1 the most
// significant) of 16 bytes at dst + (s - 1) stride holds d_s 2^(kScale - 7 s), a BF16
// value exactly, |d_s| <= 64.  Carrying the weight of a digit in its exponent costs
// nothing and puts every pair of a diagonal on one scale, 2^(2 kScale - 7 (s + t)).
//
// What bounds the kernels is the ALU pipe (16 lanes a clock and scheduler: shifts, logic,
// byte permutes), so the digits are cut by float32 additions (32 lanes a clock): x is
// rounded to the digit's grid by adding and subtracting 1.5 2^23 times the grid, three
// additions a digit.  float32 values enter that chain as they are, scaled by a power of
// two; float64 values as three pieces of their 56-bit integer (14, 21 and 21 bits, the
// lower ones balanced by a bias), each placed in a float32 mantissa by one logic operation.
template <typename T> struct Digits;
template <> struct Digits<float> {
  static constexpr int S = 5, T = 6, kScale = 3;
  // V = round(x 2^(160 - E)), |V| <= 2^34, V = sum d_s 2^(7 (5 - s))
  __device__ static void store(const float (&v)[8], int E, unsigned char* dst, int stride) {
    const bool in = E > 0 && E < 255;     // zero and subnormal groups, and Inf or NaN, give zeros
    const float sc = __uint_as_float((uint32_t)(255 - E) << 23);   // 2^(128 - E): |x| < 4
    float x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = in ? v[q] * sc : 0.f;
    take_plane<kScale - 7>(x, dst);
    take_plane<kScale - 14>(x, dst + stride);
    take_plane<kScale - 21>(x, dst + 2 * stride);
    take_plane<kScale - 28>(x, dst + 3 * stride);
    take_plane<kScale - 35>(x, dst + 4 * stride);
  }
};
template <> struct Digits<double> {
  static constexpr int S = 8, T = 9, kScale = 14;
  // V = round(x 2^(55 - E + 1022)), |V| <= 2^55, V = sum d_s 2^(7 (8 - s))
  __device__ static void store(const double (&v)[8], int E, unsigned char* dst, int stride) {
    uint32_t wl[8], wh[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int hi = __double2hiint(v[q]), lo = __double2loint(v[q]);
      const int e = (hi >> 20) & 0x7FF;
      unsigned long long m =
          ((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (uint32_t)(lo << 11);
      const int sh = e ? E - e + 8 : 64;              // zero, and subnormal (below every digit): 0
      asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(sh));   // a shift past 63 gives 0
      // 2 V + 1 + 2 (2^41 + 2^20): one bit more than V for the rounding, and the biases of
      // the two lower pieces
      const long long s = (long long)(hi >> 31);
      const long long w = ((long long)m ^ s) + ((2 * ((1ll << 41) + (1ll << 20)) + 1) - s);
      wl[q] = (uint32_t)w;
      wh[q] = (uint32_t)((unsigned long long)w >> 32);
    }
    float x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = __uint_as_float(0x4B400000u + (uint32_t)((int)wh[q] >> 11)) - 12582912.f;
    take_plane<7>(x, dst);
    store_plane(dst + stride, x);
#pragma unroll
    for (int q = 0; q < 8; ++q)   // (2^23 + u) 2^-21 - 4.5 = (u - 2^20) 2^-21
      x[q] = fmaf(__uint_as_float((__funnelshift_r(wl[q], wh[q], 22) & 0x1FFFFFu) | 0x4B000000u), pow2f(-21), -4.5f);
    take_plane<-7>(x, dst + 2 * stride);
    take_plane<-14>(x, dst + 3 * stride);
    store_plane(dst + 4 * stride, x);
#pragma unroll
    for (int q = 0; q < 8; ++q)   // (2^23 + 2 u) 2^-43 - 5 2^-22 = (u - 2^20) 2^-42
      x[q] = fmaf(__uint_as_float((wl[q] & 0x3FFFFEu) | 0x4B000000u), pow2f(-43), -5.f * pow2f(-22));
    take_plane<-28>(x, dst + 5 * stride);
    take_plane<-35>(x, dst + 6 * stride);
    store_plane(dst + 7 * stride, x);
  }
};

// The MMAs of one K-step of a sub-chunk: every digit pair (s, t) with s + t <= T into the
// accumulator of its diagonal, the kNB columns from (s + t - 2) * kNB of the allocation.
//
// The planes of the B operand follow one another at the stride of its 8-row groups, and the
// diagonals of s and consecutive t are consecutive accumulators, so that one MMA of
// N = kNB m multiplies plane s of A with m planes of B: the A plane is read from shared
// memory once for them (MMAs of N = 64 were held to a third of the tensor rate by the reads of
// their operands).  tcgen05.mma are executed in the order of issue only where they have the
// same accumulator and the same shape; others may overtake one another, and an accumulation
// or the overwriting at the start of a window would be lost.  The accumulators are therefore
// taken in fixed groups of mma_planes(S) diagonals, and every MMA that writes a group has the
// group's base and N: where a group begins before the diagonal of (s, 1), the first planes
// of B are the zero planes in front of plane 1, which add nothing.
// 12 MMAs of N = 256 for float64 digits, 3 of N = 192 and 5 of 128 for float32 digits (655362
// x 128: Gram 1030 us and 578 us; in groups of two 1099 and 613, of three float64 and four
// float32 diagonals 1072 and 599).
struct MmaOp {
  int s, t, col, n;   // plane of A, first plane of B (below 1: a zero plane), columns
};
template <int S, int T>
struct MmaPlan {
  int count = 0;
  MmaOp op[S * T] = {};
  __host__ __device__ constexpr MmaPlan() {
    constexpr int W = mma_planes(S);
    for (int s = 1; s <= S; ++s)
      for (int d = 0; d <= T - 2; d += W) {            // diagonals s + t - 2 = d .. d + m - 1
        const int m = T - 1 - d < W ? T - 1 - d : W, t = d - s + 2;
        if (t + m - 1 >= 1) op[count++] = {s, t, d * kNB, m * kNB};
      }
  }
  // every pair once and nothing else but zero planes, the first MMA of each group covering it,
  // and one base and N for all MMAs that share a column
  constexpr bool sound() const {
    int seen[S + 1][S + 1] = {};
    for (int q = 0; q < count; ++q) {
      const MmaOp& a = op[q];
      if (a.t < 1 - zero_planes(S) || a.col + a.n > (T - 1) * kNB || a.n > 256) return false;
      for (int v = 0; v < a.n / kNB; ++v) {
        const int t = a.t + v;
        if (t > S || a.s + t - 2 != a.col / kNB + v) return false;
        if (t >= 1) ++seen[a.s][t];
      }
      for (int p = 0; p < q; ++p) {
        const MmaOp& b = op[p];
        if (a.col < b.col + b.n && b.col < a.col + a.n && (a.col != b.col || a.n != b.n)) return false;
      }
      bool opens = true;                               // the first writer of its columns is plane 1
      for (int p = 0; p < q; ++p) opens = opens && op[p].col != a.col;
      if (opens != (a.s == 1)) return false;
    }
    for (int s = 1; s <= S; ++s)
      for (int t = 1; t <= S; ++t)
        if (seen[s][t] != (s + t <= T ? 1 : 0)) return false;
    return true;
  }
};
static_assert(MmaPlan<Digits<double>::S, Digits<double>::T>().sound(), "MMAs of float64 digits");
static_assert(MmaPlan<Digits<float>::S, Digits<float>::T>().sound(), "MMAs of float32 digits");

// Issues the MMAs of one sub-chunk (sB: the first zero plane of B).  first: the sub-chunk opens
// an accumulation window (plane 1 of A reaches every diagonal and overwrites it).
template <int S, int T>
__device__ __forceinline__ void issue_mmas(uint32_t tmem, uint32_t sA, uint32_t sB, bool first) {
  constexpr MmaPlan<S, T> plan;
#pragma unroll
  for (int ks = 0; ks < kKsub / 16; ++ks) {
#pragma unroll
    for (int q = 0; q < plan.count; ++q) {
      const MmaOp op = plan.op[q];
      const uint64_t ad = sdesc(sA + (op.s - 1) * kAPlane + ks * 256, 128, kKsub * 16);
      const uint64_t bd = sdesc(sB + (op.t - 1 + zero_planes(S)) * kBPlane + ks * 256, 128, kKsub * 16);
      mma_bf16(tmem + (uint32_t)op.col, ad, bd, idesc_bf16(128, op.n), (first && op.s == 1 && ks == 0) ? 0u : 1u);
    }
  }
}

// 4 consecutive TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr));
}

// Exact integers hi 2^32 + lo (lo unsigned) of the output elements: sum over the diagonals
// of A_dg 2^((T - dg) 7), A_dg the integer sum of a diagonal's digit products (at most
// 2^23): below 2^72 for float64 digits.  float32 digits (T = 6) stay below 2^51: hi is the
// sign.
struct Wide {
  long long hi;
  uint32_t lo;
};
// floor(w / 2^sh), sh >= 0
__device__ __forceinline__ void wide_sra(Wide& w, int sh) {
  if (sh == 0) return;
  if (sh < 32) {
    w.lo = __funnelshift_r(w.lo, (uint32_t)w.hi, sh);
    w.hi >>= sh;
  } else {
    w.lo = (uint32_t)(w.hi >> (sh - 32 > 63 ? 63 : sh - 32));
    w.hi = w.hi >> (sh > 63 ? 63 : sh);
  }
}
__device__ __forceinline__ void wide_add(Wide& a, const Wide& b) {
  const uint32_t l = a.lo + b.lo;
  a.hi += b.hi + (l < a.lo ? 1 : 0);
  a.lo = l;
}
// Reads the T - 1 diagonals of 4 output columns of this thread's TMEM lane and combines
// them; sc: the digits' scales, an accumulator of diagonal dg holds A_dg 2^(sc - 7 dg).
template <int T>
__device__ __forceinline__ void read_window(uint32_t taddr, int sc2, Wide (&out)[4]) {
  uint32_t v[T - 1][4];
#pragma unroll
  for (int dg = 2; dg <= T; ++dg) tmem_ld4(taddr + (uint32_t)((dg - 2) * kNB), v[dg - 2]);
  tmem_wait_ld();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int A[T - 1];
#pragma unroll
    for (int dg = 2; dg <= T; ++dg)
      A[dg - 2] = __float2int_rn(__uint_as_float(v[dg - 2][q]) * __uint_as_float((uint32_t)(127 + 7 * dg - sc2) << 23));
    // low: the last five diagonals (below 2^53), high: the others, in units of 2^32
    long long low = A[T - 2], high = 0;
#pragma unroll
    for (int dg = T - 1; dg >= (T - 4 > 2 ? T - 4 : 2); --dg) low += (long long)A[dg - 2] * (1 << ((T - dg) * 7));
#pragma unroll
    for (int dg = T - 5; dg >= 2; --dg) high += (long long)A[dg - 2] * (1 << ((T - dg) * 7 - 32));
    out[q].lo = (uint32_t)low;
    out[q].hi = high + (low >> 32);
  }
}

// v 2^e for a float64 v, by a power-of-two factor when 2^e is a normal number
__device__ __forceinline__ double scale2(double v, int e) {
  if (e >= -1022 && e <= 1023) return v * __longlong_as_double((long long)(e + 1023) << 52);
  return ldexp(v, e);
}
__device__ __forceinline__ double wide_value(const Wide& w, int e) {
  return scale2(fma((double)w.hi, 4294967296.0, (double)w.lo), e);
}

// exponent offset of the product value: x y = 2^(Ex + Gy + off) (hi 2^32 + lo)
template <typename TA, typename TB, int S, int T>
__host__ __device__ constexpr int value_offset() {
  return -Fmt<TA>::bias - Fmt<TB>::bias + 2 - 2 * (kBeta * S - 1) + (2 * S - T) * kBeta;
}

// Output value of the expansion: Z + (hi 2^32 + lo) 2^e.
template <typename TI> struct Epi;
template <> struct Epi<double> {
  // A float64 operation costs a warp 64 cycles here, so the value is brought to its 63
  // leading bits by shifts, converted once (rounded to nearest) and scaled in its exponent
  // field.
  __device__ static double value(const Wide& w, int e) {
    const int n = min(__clzll(w.hi ^ (w.hi >> 63)) - 1, 32);   // shift that keeps the sign
    const long long v =
        n == 0 ? w.hi : (long long)(((unsigned long long)w.hi << n) | ((unsigned long long)w.lo >> (32 - n)));
    if (v == 0) return 0.0;
    const double d = __ll2double_rn(v);
    const int f = e + 32 - n, hi = __double2hiint(d), ef = ((hi >> 20) & 0x7FF) + f;
    if (ef < 1 || ef > 2046) return scale2(d, f);
    return __hiloint2double(hi + (f << 20), __double2loint(d));
  }
};
template <> struct Epi<float> {
  __device__ static float value(const Wide& w, int e) {
    const float v = (float)(long long)(((unsigned long long)w.hi << 32) | w.lo);   // below 2^51
    if (e >= -126 && e <= 127) return v * __int_as_float((e + 127) << 23);
    return ldexpf(v, e);
  }
};

// Launch controls: the limit of every bounded wait, and (timeout self-tests only) an
// MMA warp that issues nothing, so that the workers' waits for commits expire.
struct TcCtl {
  long long wait_cycles;
  int no_mma;
};

struct TcShared {
  long long wait_limit;
  int no_mma;
  uint64_t bar[2];    // stage b free again: the commit of its MMAs (one arrival)
  uint64_t full[2];   // stage b holds digits: one arrival per worker warp
  uint32_t tmem_slot;
  int abort_flag;
  // exponents of the 128 A rows (Gram: columns of X; expand: rows of X) and of the kNB B
  // rows (Gram: columns of Y; expand: columns of Yx), windows or tiles in turn (the scan
  // warps write the next one while the readback of the last one may still run); Gram: the
  // running exponents of the B rows after each window
  int exA[4][128], exB[4][kNB], run[4][kNB];
};

template <int S>
__device__ __forceinline__ unsigned char* stage_ptr(unsigned char* smem, int b) {
  return smem + b * stage_bytes(S);
}

// TMEM columns: one kNB-wide accumulator per diagonal, rounded up to a power of two.
template <int T>
__host__ __device__ constexpr uint32_t tmem_cols() {
  return (T - 1) * kNB <= 32 ? 32 : (T - 1) * kNB <= 64 ? 64 : (T - 1) * kNB <= 128 ? 128 : (T - 1) * kNB <= 256 ? 256 : 512;
}

// barriers of the worker warps only, and of the worker and scan warps (the MMA warp takes
// part in neither)
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory"); }
__device__ __forceinline__ void scan_sync() { asm volatile("bar.sync 3, %0;" ::"n"(32 * kScanWarps) : "memory"); }
// (returns to all of them alike whether one of them had seen the abort flag)
__device__ __forceinline__ bool workers_scan_sync(const int* abort_flag) {
  const int seen = *reinterpret_cast<const volatile int*>(abort_flag);
  int any;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %2, 0;\nbar.red.or.pred q, 2, %1, p;\nselp.b32 %0, 1, 0, q;\n}\n"
      : "=r"(any)
      : "n"(kWorkers + 32 * kScanWarps), "r"(seen)
      : "memory");
  return any != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(su32(bar)) : "memory");
}

template <int T>
__device__ __forceinline__ void tc_setup(TcShared& sh, unsigned char* smem, int bytes, const TcCtl& ctl) {
  const int tid = threadIdx.x;
  for (int q = tid; q < bytes / 16; q += blockDim.x) reinterpret_cast<uint4*>(smem)[q] = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    sh.wait_limit = ctl.wait_cycles;
    sh.no_mma = ctl.no_mma;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&sh.bar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&sh.bar[1])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&sh.full[0])), "n"(kWorkers / 32));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&sh.full[1])), "n"(kWorkers / 32));
    sh.abort_flag = 0;
  }
  if ((tid >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sh.tmem_slot)),
                 "r"(tmem_cols<T>()));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
}

// End of a tensor-core kernel, reached by every thread.  The issuing thread first
// waits (bounded) for the last commit of each stage, so that no MMA is in flight when
// the tensor memory is freed (after a timed-out wait the MMAs may still run).  *err: bit 0 a
// wait expired, bit 1 the workers and scan warps left their loops for it (left).
template <int T>
__device__ __forceinline__ void tc_teardown(TcShared& sh, int issued, int* err, bool left = false) {
  if (threadIdx.x == kWorkers) {
    for (int b = 0; b < 2; ++b) {
      const int uses = (issued - b + 1) / 2;   // commits made on stage b
      if (uses > 0 && !mbar_wait(&sh.bar[b], (uint32_t)((uses - 1) & 1), sh.wait_limit)) atomicExch(&sh.abort_flag, 1);
    }
  }
  fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem_slot), "r"(tmem_cols<T>()));
  }
  if (sh.abort_flag && threadIdx.x == 0) atomicOr(err, left ? 3 : 1);
}

// Waits (every worker) for the commit of sub-chunk gi; raises the shared abort flag
// on expiry.  Workers read the flag only right after a worker barrier, so that they
// leave their loops together.
__device__ __forceinline__ void wait_sub(TcShared& sh, int gi) {
  if (!mbar_wait(&sh.bar[gi & 1], (uint32_t)((gi >> 1) & 1), sh.wait_limit)) atomicExch(&sh.abort_flag, 1);
}

// The MMA warp's part for sub-chunk g (sc: its index in the accumulation window):
// lane 0 waits for the workers' digits of stage g & 1, issues the MMAs and commits
// them to the stage's free barrier.  Returns false (warp-uniform) when the wait expired.
template <int S, int T>
__device__ __forceinline__ bool mma_step(TcShared& sh, unsigned char* smem, uint32_t tmem, int g, int sc) {
  const int lane = threadIdx.x & 31;
  const int b = g & 1;
  int ok = 1;
  if (lane == 0) ok = mbar_wait(&sh.full[b], (uint32_t)((g >> 1) & 1), sh.wait_limit) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) {
    if (lane == 0) atomicExch(&sh.abort_flag, 1);
    return false;
  }
  if (lane == 0 && !sh.no_mma) {
    fence_after();
    const uint32_t sA = su32(stage_ptr<S>(smem, b));
    issue_mmas<S, T>(tmem, sA, sA + S * kAPlane, sc == 0);   // (the zero planes follow the planes of A)
    mma_commit(&sh.bar[b]);
  }
  __syncwarp();
  return true;
}

// A worker warp hands stage b to the MMA warp: every lane's digit stores made visible
// to the tensor cores' (async) proxy, then one arrival for the warp.
__device__ __forceinline__ void hand_over(TcShared& sh, int b) {
  fence_async_smem();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&sh.full[b]);
}

// Brings rows [ra, rb) of a block, `bytes` of each from p on, to L2 (a warp; no register waits
// for the data, unlike for loads far ahead).
__device__ __forceinline__ void prefetch_rows(const void* p, size_t stride, int bytes, int ra, int rb, int first,
                                              int step) {
  const int lines = (bytes + 127) / 128;
  const int total = (rb - ra) * lines;
  for (int q = first; q < total; q += step) {
    const char* a = static_cast<const char*>(p) + (size_t)(ra + q / lines) * stride + (size_t)(q % lines) * 128;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
  }
}

// ------------------------------------------------------------ Gram kernel -----
// blockIdx.x: row part [r0, r1); blockIdx.y: block of kNB columns of Y.
// partial[part][i * k + j] = (X[r0:r1, i])^T Y[r0:r1, j] for i < k and j in the block.
// Warps 0-15 form the digits of each 32-row sub-chunk and read the window sums back;
// warp 16 issues the MMAs.  A thread owns one column of X and 8 rows of the sub-chunk (a
// 16-byte store a digit, free of bank conflicts), and every other sub-chunk also 8 rows of
// one column of Y, so that the two halves of the warps take turns with the longer part.
// The exponents of the next window are gathered while the digits of the current one are
// formed (those loads bring the block from DRAM, the digits' loads then find it in L2), and
// a window's sums are read back after the digits of the next window's first sub-chunk are
// stored, so that the MMAs in flight are not waited for at once.
template <typename TI>
__global__ void __launch_bounds__(kTcThreads, 1)
gram_tc_kernel(const TI* __restrict__ X, const TI* __restrict__ Y, int n, int k, int ld, int rows_per_part,
               double* __restrict__ partial, int vec, int* err, TcCtl ctl) {
  constexpr int S = Digits<TI>::S, T = Digits<TI>::T;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ TcShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int jb = blockIdx.y * kNB;
  const int r0 = blockIdx.x * rows_per_part;
  const int r1 = min(n, r0 + rows_per_part);
  tc_setup<T>(sh, smem, 2 * stage_bytes(S), ctl);
  const uint32_t tmem = sh.tmem_slot;
  if (warp == kMmaWarp) {
    int g = 0;
    bool ok = true;
    for (int w0 = r0; w0 < r1 && ok; w0 += kWindow) {
      const int nsub = (min(r1, w0 + kWindow) - w0 + kKsub - 1) / kKsub;
      for (int sc = 0; sc < nsub && ok; ++sc) {
        ok = mma_step<S, T>(sh, smem, tmem, g, sc);
        if (ok) ++g;
      }
    }
    tc_teardown<T>(sh, sh.no_mma ? 0 : g, err);
    return;
  }
  if (warp >= kScan0) {
    // Exponents of the windows after the first (the workers gather those), a window ahead:
    // a lane takes 16 bytes of a row of [X | the block of Y] (float32: the lanes of a warp
    // part take every other row), 16 rows in flight, and keeps the largest magnitude word of
    // each column.  The rows are brought to L2 kAhead rows before.  8-byte (4-byte) loads
    // from DRAM took 1.1 ms (0.9 ms) over 655362 x 128, longer than everything else.
    constexpr int kAhead = 64, kVals = 16 / (int)sizeof(TI);
    constexpr int kFly = 16;
    constexpr int kLanes = (128 + kNB) / kVals, kSplit = 32 * kScanWarps / kLanes;
    static_assert(kLanes * kSplit == 32 * kScanWarps, "the lanes of the scan warps cover [X | Y]");
    const int st = tid - 32 * kScan0, part = st / kLanes;
    const int c0 = (st % kLanes) * kVals, cy0 = c0 - 128;
    const bool in = cy0 < 0 ? c0 < k : jb + cy0 < k;
    const int cols = cy0 < 0 ? k - c0 : k - jb - cy0;     // valid columns from c0 on
    const TI* p = cy0 < 0 ? X + c0 : Y + jb + cy0;
    const size_t stride = (size_t)ld * sizeof(TI);
    // prefetch: 16 lanes a row, the 128-byte lines of X (at most 8) and of the block of Y (4)
    const int pl = st & 15, pbytes = (pl < 8 ? min(128, k) : min(kNB, k - jb)) * (int)sizeof(TI);
    const int poff = (pl < 8 ? pl : pl - 8) * 128;
    const char* pp = reinterpret_cast<const char*>(pl < 8 ? X : Y + jb) + poff;
    const bool pin = poff < pbytes;
    auto ahead = [&](int ra, int rb) {
      rb = min(rb, r1);
      if (pin)
        for (int r = ra + (st >> 4); r < rb; r += 32 * kScanWarps / 16)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(pp + (size_t)r * stride));
    };
    ahead(r0, r0 + kWindow + kAhead);
    workers_scan_sync(&sh.abort_flag);
    int run[kVals];
#pragma unroll
    for (int v = 0; v < kVals; ++v) run[v] = (cy0 >= 0 && part == 0) ? sh.exB[0][cy0 + v] : 0;
    int w = 0;
    for (int w0 = r0; w0 < r1; w0 += kWindow, ++w) {
      const int n1 = min(r1, w0 + 2 * kWindow), nx = (w + 1) & 3;
      uint32_t m[kVals];
#pragma unroll
      for (int v = 0; v < kVals; ++v) m[v] = 0u;
      for (int r = w0 + kWindow; r < n1; r += kFly * kSplit) {
        ahead(r + kAhead, r + kAhead + kFly * kSplit);
        uint32_t x[kFly][kVals];
#pragma unroll
        for (int q = 0; q < kFly; ++q) {
          const int rr = r + part + q * kSplit;
#pragma unroll
          for (int v = 0; v < kVals; ++v) x[q][v] = 0u;
          if (in && rr < n1) Fmt<TI>::words(p + (size_t)rr * ld, cols, vec != 0, x[q]);
        }
#pragma unroll
        for (int q = 0; q < kFly; ++q)
#pragma unroll
          for (int v = 0; v < kVals; ++v) m[v] = max(m[v], x[q][v] & 0x7fffffffu);
      }
      // the parts' maxima meet in shared memory (kSplit > 1: through atomics on a zeroed slot)
      int e[kVals];
#pragma unroll
      for (int v = 0; v < kVals; ++v) e[v] = v < cols ? Fmt<TI>::expo_of(m[v]) : 0;
      if constexpr (kSplit == 1) {
#pragma unroll
        for (int v = 0; v < kVals; ++v)
          if (cy0 < 0) sh.exA[nx][c0 + v] = e[v]; else sh.exB[nx][cy0 + v] = e[v];
      } else {
        int* slot = cy0 < 0 ? &sh.exA[nx][c0] : &sh.exB[nx][cy0];
        if (part == 0)
#pragma unroll
          for (int v = 0; v < kVals; ++v) slot[v] = e[v];
        scan_sync();
        if (part != 0)
#pragma unroll
          for (int v = 0; v < kVals; ++v) atomicMax(slot + v, e[v]);
        scan_sync();
#pragma unroll
        for (int v = 0; v < kVals; ++v) e[v] = slot[v];
      }
      if (cy0 >= 0 && part == 0)
#pragma unroll
        for (int v = 0; v < kVals; ++v) {
          run[v] = max(run[v], e[v]);
          sh.run[nx][cy0 + v] = run[v];
        }
      if (workers_scan_sync(&sh.abort_flag)) break;
    }
    tc_teardown<T>(sh, 0, err);
    return;
  }
  // digit ownership: column cx of X, rows 8 kx .. 8 kx + 7 of a sub-chunk; column jb + cy of
  // Y, rows 8 ky .. (sub-chunks of the parity of the warp's half)
  const int cx = tid & 127, kx = tid >> 7, cy = tid & (kNB - 1), ky = (tid >> 6) & 3, half = tid >> 8;
  const bool has_x = cx < k, has_y = jb + cy < k;
  // readback ownership: TMEM lane i = row of the output block, 16 columns
  const int i_out = (warp & 3) * 32 + lane;
  const int c_base = (warp >> 2) * 16;
  const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c_base;
  Wide R[16];               // running sums of the 16 outputs of this thread
#pragma unroll
  for (int q = 0; q < 16; ++q) R[q] = {0, 0u};
  int e_run = 0;
  // running sums += window w (its MMAs complete), aligned to the larger exponents
  auto readback = [&](int w) {
    const int eA = sh.exA[w & 3][i_out];
    const int newE = max(e_run, eA);
    const int dR = newE - e_run, dW = newE - eA;
    e_run = newE;
    const int* exB = sh.exB[w & 3];
    const int* now = sh.run[w & 3];
    const int* was = sh.run[(w + 3) & 3];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      Wide W[4];
      read_window<T>(tlane + ch * 4, 2 * Digits<TI>::kScale, W);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int jj = c_base + ch * 4 + q;
        wide_sra(R[ch * 4 + q], dR + now[jj] - was[jj]);
        wide_sra(W[q], dW + now[jj] - exB[jj]);
        wide_add(R[ch * 4 + q], W[q]);
      }
    }
    fence_before();
  };
  if (tid < kNB) {
    sh.run[3][tid] = 0;
    sh.exB[0][tid] = 0;
  }
  if (tid < 128) sh.exA[0][tid] = 0;
  workers_sync();
  {
    // exponents of the first window
    const int w1 = min(r1, r0 + kWindow);
    int m = 0, mb = 0;
    if (has_x) {
#pragma unroll 8
      for (int r = r0 + kx; r < w1; r += kWorkers / 128) m = max(m, Fmt<TI>::expo(X[(size_t)r * ld + cx]));
    }
    if (has_y) {
#pragma unroll 8
      for (int r = r0 + (tid / kNB); r < w1; r += kWorkers / kNB) mb = max(mb, Fmt<TI>::expo(Y[(size_t)r * ld + jb + cy]));
    }
    if (m) atomicMax(&sh.exA[0][cx], m);
    if (mb) atomicMax(&sh.exB[0][cy], mb);
  }
  workers_scan_sync(&sh.abort_flag);
  if (tid < kNB) sh.run[0][tid] = sh.exB[0][tid];
  int g = 0, w = 0;
  bool left = false;        // the same in every worker: the flag itself may rise at any time
  for (int w0 = r0; w0 < r1; w0 += kWindow, ++w) {
    const int w1 = min(r1, w0 + kWindow);
    const int nsub = (w1 - w0 + kKsub - 1) / kKsub;
    const int EA = sh.exA[w & 3][cx], EB = sh.exB[w & 3][cy];
    for (int sc = 0; sc < nsub; ++sc, ++g) {
      const int b = g & 1;
      const bool do_y = has_y && (g & 1) == half;
      const int rb = w0 + sc * kKsub;
      TI vx[8], vy[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = rb + kx * 8 + q;
        vx[q] = (has_x && r < r1) ? X[(size_t)r * ld + cx] : TI(0);
      }
      if (do_y) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int r = rb + ky * 8 + q;
          vy[q] = r < r1 ? Y[(size_t)r * ld + jb + cy] : TI(0);
        }
      }
      if (g >= 2) wait_sub(sh, g - 2);
      unsigned char* st = stage_ptr<S>(smem, b);
      if (has_x) Digits<TI>::store(vx, EA, st + cm_off(cx, kx * 8), kAPlane);
      if (do_y) Digits<TI>::store(vy, EB, st + b_offset(S) + cm_off(cy, ky * 8), kBPlane);
      if (sc == 0 && w > 0) {
        wait_sub(sh, g - 1);
        __syncwarp();
        fence_after();
        readback(w - 1);
      }
      hand_over(sh, b);
    }
    left = workers_scan_sync(&sh.abort_flag);        // the exponents of the next window are complete
    if (left) break;
  }
  if (w > 0 && !left) {
    wait_sub(sh, g - 1);
    __syncwarp();
    fence_after();
    readback(w - 1);
  }
  workers_sync();
  if (!sh.abort_flag && i_out < k) {
    constexpr int off = value_offset<TI, TI, S, T>();
    const int* run = sh.run[(w + 3) & 3];
    double* out = partial + (size_t)blockIdx.x * k * k + (size_t)i_out * k;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int j = jb + c_base + q;
      if (j < k)
        out[j] = (e_run == Fmt<TI>::emax || run[c_base + q] == Fmt<TI>::emax)
                     ? __longlong_as_double(0x7FF8000000000000ll)
                     : wide_value(R[q], e_run + run[c_base + q] + off);
    }
  }
  tc_teardown<T>(sh, 0, err, left);
}

// ------------------------------------------------------------ expand ----------
// 8 float64 values of a column of Yx as digits beside those of blocks of type TI: for
// float32 blocks the 5 digits of V = round(x 2^(34 - E + 1022)), in two pieces of 21 and 14
// bits.
template <typename TI>
__device__ __forceinline__ void store_yx(const double (&v)[8], int E, unsigned char* dst) {
  if constexpr (sizeof(TI) == 8) {
    Digits<double>::store(v, E, dst, kBPlane);
  } else {
    float hi[8], lo[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v[q]);
      const int e = (int)((b >> 52) & 0x7FF);
      unsigned long long m = (b << 11) | 0x8000000000000000ull;
      const int sh = e ? E - e + 29 : 64;                       // 35 bits: one more for the rounding
      asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(sh));
      const long long V = (long long)((m + 1) >> 1);
      const long long w = ((b >> 63) ? -V : V) + (1ll << 13);
      hi[q] = (float)(int)(w >> 14) * pow2f(-18);
      lo[q] = (float)((int)(w & 0x3FFF) - (1 << 13)) * pow2f(-32);
    }
    take_plane<-4>(hi, dst);
    take_plane<-11>(hi, dst + kBPlane);
    store_plane(dst + 2 * kBPlane, hi);
    take_plane<-25>(lo, dst + 3 * kBPlane);
    store_plane(dst + 4 * kBPlane, lo);
  }
}

// Digits of the B operand of the expansion, Yx (k x k, float64, row stride ldy):
// B[j][q] = Yx[q][j], one CTA per block of kNB columns j and sub-chunk of kKsub values q,
// S planes in the shared-memory layout; gexp[j] = exponent of column j.
constexpr int kPrepThreads = 4 * kNB;
template <typename TI>
__global__ void __launch_bounds__(kPrepThreads)
expand_prep_kernel(const double* __restrict__ Yx, int k, int ldy, unsigned char* __restrict__ dig,
                   int* __restrict__ gexp) {
  constexpr int S = Digits<TI>::S;
  __shared__ int ex[kNB];
  const int j = threadIdx.x % kNB, part = threadIdx.x / kNB, col = blockIdx.x * kNB + j, sc = blockIdx.y;
  if (threadIdx.x < kNB) ex[j] = 0;
  __syncthreads();
  int m = 0;
  if (col < k) {
#pragma unroll 8
    for (int q = part; q < k; q += kPrepThreads / kNB) m = max(m, Fmt<double>::expo(Yx[(size_t)q * ldy + col]));
  }
  if (m) atomicMax(&ex[j], m);
  __syncthreads();
  if (sc == 0 && threadIdx.x < kNB) gexp[col] = ex[j];
  double v[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int q = sc * kKsub + part * 8 + t;
    v[t] = (col < k && q < k) ? Yx[(size_t)q * ldy + col] : 0.0;
  }
  store_yx<TI>(v, ex[j], dig + ((size_t)blockIdx.x * gridDim.y + sc) * S * kBPlane + cm_off(j, part * 8));
}

// 4 (8) consecutive values from index i of a block, `left` of them inside the row: 16-byte
// accesses when vec (base and row stride multiples of 16 bytes), zeros outside
template <int N>
__device__ __forceinline__ void ld_vals(const double* p, size_t i, int left, bool vec, double (&v)[N]) {
  if (vec) {
#pragma unroll
    for (int q = 0; q < N; q += 2) {
      double2 t = make_double2(0.0, 0.0);
      if (q < left) t = *reinterpret_cast<const double2*>(p + i + q);
      v[q] = t.x;
      v[q + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = q < left ? p[i + q] : 0.0;
  }
}
template <int N>
__device__ __forceinline__ void ld_vals(const float* p, size_t i, int left, bool vec, float (&v)[N]) {
  if (vec) {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q < left) t = *reinterpret_cast<const float4*>(p + i + q);
      v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = q < left ? p[i + q] : 0.f;
  }
}
__device__ __forceinline__ void st_vals(double* p, size_t i, int left, bool vec, const double (&v)[4]) {
  if (vec) {
    if (left > 0) *reinterpret_cast<double2*>(p + i) = make_double2(v[0], v[1]);
    if (left > 2) *reinterpret_cast<double2*>(p + i + 2) = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < left) p[i + q] = v[q];
  }
}
__device__ __forceinline__ void st_vals(float* p, size_t i, int left, bool vec, const float (&v)[4]) {
  if (vec) {
    if (left > 0) *reinterpret_cast<float4*>(p + i) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < left) p[i + q] = v[q];
  }
}

// U[r][j] = Z[r][j] + sum_q X[r][q] Yx[q][j]: persistent CTAs take 128-row tiles in turn,
// and the kNB-column blocks of a tile one after the other (the X tile is then found in
// L1 and L2).  Warps 0-15 form the X digits of each 32-value sub-chunk (8 values of a row a
// thread), copy the prepared Yx digits and write U; warp 16 issues the MMAs.  As in the
// Gram kernel, the row exponents of the next tile are gathered during the current one, and
// a block's sums are read back after the digits of the next block's first sub-chunk.
template <typename TI>
__global__ void __launch_bounds__(kTcThreads, 1)
expand_tc_kernel(const TI* __restrict__ Z, const TI* __restrict__ X, const unsigned char* __restrict__ dig,
                 const int* __restrict__ gexp, int n, int k, int ld, int nsub, int njb, TI* __restrict__ U,
                 int vec, int* err, TcCtl ctl) {
  constexpr int S = Digits<TI>::S, T = Digits<TI>::T;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ TcShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  tc_setup<T>(sh, smem, 2 * stage_bytes(S), ctl);
  const uint32_t tmem = sh.tmem_slot;
  const int ntiles = (n + 127) / 128;
  // this CTA's column blocks: all, or (gridDim.y = njb) one
  const int jb0 = gridDim.y > 1 ? blockIdx.y : 0, jb1 = gridDim.y > 1 ? jb0 + 1 : njb;
  if (warp == kMmaWarp) {
    int g = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x)
      for (int u = 0; u < (jb1 - jb0) * nsub && ok; ++u) {
        ok = mma_step<S, T>(sh, smem, tmem, g, u % nsub);
        if (ok) ++g;
      }
    tc_teardown<T>(sh, sh.no_mma ? 0 : g, err);
    return;
  }
  if (warp >= kScan0) {
    // row exponents of the next tile, 8 rows of a warp in flight; the rows of X after it and
    // those of Z are brought to L2 meanwhile
    constexpr int kVals = 16 / (int)sizeof(TI);
    const int sw = warp - kScan0;
    const size_t stride = (size_t)ld * sizeof(TI);
    auto ahead = [&](const TI* p, int tl) {
      if (p && tl < ntiles)
        prefetch_rows(p, stride, k * (int)sizeof(TI), tl * 128, min(n, tl * 128 + 128), sw * 32 + lane, 32 * kScanWarps);
    };
    ahead(X, blockIdx.x + gridDim.x);
    int t = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++t) {
      const int base = (tile + (int)gridDim.x) * 128;
      ahead(Z, tile);
      ahead(X, tile + 2 * gridDim.x);
      for (int a0 = sw * 8; a0 < 128; a0 += 8 * kScanWarps) {
        uint32_t m[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) m[q] = 0u;
        if (base + a0 < n)
          for (int c = lane * kVals; c < k; c += 64 * kVals) {
            uint32_t x[16][kVals], mask[2][kVals];     // magnitudes of the columns below k
#pragma unroll
            for (int v = 0; v < kVals; ++v) {
              mask[0][v] = c + v < k ? 0x7fffffffu : 0u;
              mask[1][v] = c + 32 * kVals + v < k ? 0x7fffffffu : 0u;
            }
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const int cq = c + (q & 1) * 32 * kVals, r = base + a0 + (q >> 1);
#pragma unroll
              for (int v = 0; v < kVals; ++v) x[q][v] = 0u;
              if (r < n && cq < k) Fmt<TI>::words(X + (size_t)r * ld + cq, k - cq, vec != 0, x[q]);
            }
#pragma unroll
            for (int q = 0; q < 16; ++q)
#pragma unroll
              for (int v = 0; v < kVals; ++v) m[q >> 1] = max(m[q >> 1], x[q][v] & mask[q & 1][v]);
          }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int e = Fmt<TI>::expo_of(__reduce_max_sync(0xffffffffu, m[q]));
          if (lane == 0) sh.exA[(t + 1) & 3][a0 + q] = e;
        }
      }
      if (workers_scan_sync(&sh.abort_flag)) break;
    }
    tc_teardown<T>(sh, 0, err);
    return;
  }
  const int i_out = (warp & 3) * 32 + lane;
  const int c_base = (warp >> 2) * 16;
  const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c_base;
  // digit ownership: row rl of the tile, values 8 kg .. 8 kg + 7 of a sub-chunk
  const int rl = tid >> 2, kg = tid & 3;
  for (int q = tid; q < njb * kNB; q += kWorkers) sh.exB[q / kNB][q % kNB] = gexp[q];
  auto row_max = [&](int m) {        // over the 4 lanes of a row
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    return max(m, __shfl_xor_sync(0xffffffffu, m, 2));
  };
  auto expo8 = [&](int r, int q0) {  // largest exponent of 8 values of row r
    int m = 0;
    if (r < n && q0 < k) {
      TI v[8];
      ld_vals(X, (size_t)r * ld + q0, ld - q0, vec != 0, v);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q0 + q < k) m = max(m, Fmt<TI>::expo(v[q]));
    }
    return m;
  };
  {
    int m = 0;
    for (int sc = 0; sc < nsub; ++sc) m = max(m, expo8(blockIdx.x * 128 + rl, sc * kKsub + kg * 8));
    m = row_max(m);
    if (kg == 0) sh.exA[0][rl] = m;
  }
  workers_sync();
  // the outputs of column block jbi of tile t (its MMAs complete)
  auto readback = [&](int t, int tile, int jbi) {
    constexpr int off = value_offset<TI, double, S, T>();
    const int r = tile * 128 + i_out, jb = jbi * kNB;
    const int eA = sh.exA[t & 3][i_out];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      const int j0 = jb + c_base + ch * 4;
      const size_t idx = (size_t)r * ld + j0;
      TI z[4] = {TI(0), TI(0), TI(0), TI(0)};
      if (Z && r < n) ld_vals(Z, idx, ld - j0, vec != 0, z);
      Wide W[4];
      read_window<T>(tlane + ch * 4, 2 * Digits<TI>::kScale, W);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int eB = sh.exB[jbi][c_base + ch * 4 + q];
        if (j0 + q < k) {
          const TI v = Epi<TI>::value(W[q], eA + eB + off);
          z[q] = (eA == Fmt<TI>::emax || eB == Fmt<double>::emax) ? (TI)__longlong_as_double(0x7FF8000000000000ll)
                                                                 : (Z ? v + z[q] : v);
        }
      }
      if (r < n) st_vals(U, idx, ld - j0, vec != 0, z);
    }
    fence_before();
  };
  int g = 0, t = 0, ptile = -1, pjb = 0;     // the block whose sums are still in tensor memory
  bool left = false;                         // the same in every worker, as in the Gram kernel
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++t) {
    const int row = tile * 128 + rl;
    const int E = sh.exA[t & 3][rl];
    for (int jbi = jb0; jbi < jb1; ++jbi) {
      for (int sc = 0; sc < nsub; ++sc, ++g) {
        const int b = g & 1, q0 = sc * kKsub + kg * 8;
        TI v[8];
        if (row < n && q0 < k) {
          ld_vals(X, (size_t)row * ld + q0, ld - q0, vec != 0, v);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (q0 + q >= k) v[q] = TI(0);
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = TI(0);
        }
        const uint4* src = reinterpret_cast<const uint4*>(dig + ((size_t)jbi * nsub + sc) * S * kBPlane);
        constexpr int NC = (S * kBPlane / 16 + kWorkers - 1) / kWorkers;
        uint4 yd[NC];
#pragma unroll
        for (int q = 0; q < NC; ++q)
          if (tid + q * kWorkers < S * kBPlane / 16) yd[q] = __ldg(src + tid + q * kWorkers);
        if (g >= 2) wait_sub(sh, g - 2);
        unsigned char* st = stage_ptr<S>(smem, b);
        uint4* dst = reinterpret_cast<uint4*>(st + b_offset(S));
#pragma unroll
        for (int q = 0; q < NC; ++q)
          if (tid + q * kWorkers < S * kBPlane / 16) dst[tid + q * kWorkers] = yd[q];
        Digits<TI>::store(v, E, st + cm_off(rl, kg * 8), kAPlane);
        if (sc == 0 && ptile >= 0) {
          wait_sub(sh, g - 1);
          __syncwarp();
          fence_after();
          readback(jbi == jb0 ? t - 1 : t, ptile, pjb);
        }
        hand_over(sh, b);
      }
      ptile = tile;
      pjb = jbi;
    }
    left = workers_scan_sync(&sh.abort_flag);        // the exponents of the next tile are complete
    if (left) break;
  }
  if (ptile >= 0 && !left) {
    wait_sub(sh, g - 1);
    __syncwarp();
    fence_after();
    readback(t - 1, ptile, pjb);
  }
  workers_sync();
  tc_teardown<T>(sh, 0, err, left);
}

int num_sms() {
  static int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 152;
  }();
  return n;
}

}  // namespace

// Row parts of a Gram: one CTA per SM (over the column blocks), of at least kMinPart rows,
// so that a small block is spread over the SMs (a part may be shorter than a window):
// 2562 x 32 in 11 parts of 256 rows took 58 us, in 41 of 64 rows 32 us.
constexpr int kMinPart = 64;
int gram_tc_parts(int n, int k) {
  const int njb = (k + kNB - 1) / kNB;
  int parts = std::max(1, std::min((n + kMinPart - 1) / kMinPart, num_sms() / njb));
  // at most 127 windows per part (headroom of the int64 window sums)
  parts = std::max(parts, (n + 127 * kWindow - 1) / (127 * kWindow));
  return parts;
}

size_t expand_tc_scratch_bytes(int k) {
  const int njb = (k + kNB - 1) / kNB, nsub = (k + kKsub - 1) / kKsub;
  return (size_t)njb * nsub * Digits<double>::S * kBPlane + sizeof(int) * njb * kNB + 256;
}

namespace {
// blocks whose rows start on 16-byte boundaries take 16-byte accesses, others one value each
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <typename TI>
void gram_tc_launch(const TI* X, const TI* Y, int n, int k, int ld, double* G, double* partial, int nparts,
                    int* err, cudaStream_t s, bool sym, TcCtl ctl) {
  if (k > kTcMaxK) fail(BMG_ERR_INVALID_ARG, "gram_tc: k > 128");
  constexpr int S = Digits<TI>::S;
  const int njb = (k + kNB - 1) / kNB;
  // whole windows when a part holds several, else whole sub-chunks
  int rows = (n + nparts - 1) / nparts;
  const int unit = rows >= kWindow ? kWindow : kKsub;
  rows = (rows + unit - 1) / unit * unit;
  const int parts = (n + rows - 1) / rows;
  const int smem = 2 * stage_bytes(S);
  check_cuda(cudaFuncSetAttribute(gram_tc_kernel<TI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
             "cudaFuncSetAttribute(gram_tc_kernel)");
  const int vec = aligned16(X) && aligned16(Y) && (size_t)ld * sizeof(TI) % 16 == 0;
  prof_begin(KC_GRAM, s);
  gram_tc_kernel<TI><<<dim3(parts, njb), kTcThreads, smem, s>>>(X, Y, n, k, ld, rows, partial, vec, err, ctl);
  check_launch("gram_tc_kernel");
  gram_reduce(partial, parts, k, G, sym, s);
  prof_end(KC_GRAM, s, 2.0 * sizeof(TI) * n * ld + 16.0 * parts * k * k + 8.0 * k * k, 2.0 * n * k * k);
}
}  // namespace

template <typename TI>
void gram_tc(const TI* X, const TI* Y, int n, int k, int ld, double* G, double* partial, int nparts, int* err,
             cudaStream_t s, bool sym) {
  gram_tc_launch<TI>(X, Y, n, k, ld, G, partial, nparts, err, s, sym, TcCtl{kWaitCycles, 0});
}

namespace {
template <typename TI>
void expand_tc_launch(const TI* Zf, const TI* X, const double* Yx, int n, int k, int ld, int ldy, TI* U,
                      unsigned char* scratch, int* err, cudaStream_t s, int ctas, TcCtl ctl) {
  if (k > kTcMaxK) fail(BMG_ERR_INVALID_ARG, "expand_tc: k > 128");
  constexpr int S = Digits<TI>::S;
  const int njb = (k + kNB - 1) / kNB, nsub = (k + kKsub - 1) / kKsub;
  int* gexp = reinterpret_cast<int*>(scratch + (size_t)njb * nsub * Digits<double>::S * kBPlane);
  const int smem = 2 * stage_bytes(S);
  check_cuda(cudaFuncSetAttribute(expand_tc_kernel<TI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
             "cudaFuncSetAttribute(expand_tc_kernel)");
  // few tiles: a CTA per tile and column block (twice the SMs at work); many: the blocks of
  // a tile in one CTA, which then reads the X tile from DRAM and forms its exponents once
  const int ntiles = (n + 127) / 128;
  const dim3 grid(std::min(ntiles, ctas), ntiles * njb <= ctas ? njb : 1);
  const int vec = aligned16(X) && aligned16(U) && aligned16(Zf) && (size_t)ld * sizeof(TI) % 16 == 0;
  prof_begin(KC_EXPAND, s);
  expand_prep_kernel<TI><<<dim3(njb, nsub), kPrepThreads, 0, s>>>(Yx, k, ldy, scratch, gexp);
  check_launch("expand_prep_kernel");
  expand_tc_kernel<TI><<<grid, kTcThreads, smem, s>>>(Zf, X, scratch, gexp, n, k, ld, nsub, njb, U, vec, err, ctl);
  check_launch("expand_tc_kernel");
  expand_pad(Zf, n, njb * kNB, ld, U, s);
  prof_end(KC_EXPAND, s, 3.0 * sizeof(TI) * n * ld + 8.0 * k * k, 2.0 * n * k * k);
}
}  // namespace

template <typename TI>
void expand_tc(const TI* Zf, const TI* X, const double* Yx, int n, int k, int ld, int ldy, TI* U,
               unsigned char* scratch, int* err, cudaStream_t s) {
  expand_tc_launch<TI>(Zf, X, Yx, n, k, ld, ldy, U, scratch, err, s, num_sms(), TcCtl{kWaitCycles, 0});
}

// The bounded waits of the tensor-core kernels, made to run out: float64 products of zero
// 4096 x 64 blocks whose MMA warp issues nothing, with waits of about 1 ms.  A part of the Gram
// has four windows of eight sub-chunks and a CTA of the expansion eight tiles of two, so that
// the waits for a stage in use expire inside the loops and the warps leave these together; the
// kernels must raise both bits of *err, free their tensor memory and return.
// partial: kTcSelftestParts * 64^2 doubles.
void gram_tc_timeout_selftest(const double* X, double* G, double* partial, int* err, cudaStream_t s) {
  gram_tc_launch<double>(X, X, 4096, 64, 64, G, partial, kTcSelftestParts, err, s, true, TcCtl{2000000LL, 1});
}
void expand_tc_timeout_selftest(const double* X, const double* Yx, double* U, unsigned char* scratch, int* err,
                                cudaStream_t s) {
  expand_tc_launch<double>(nullptr, X, Yx, 4096, 64, 64, 64, U, scratch, err, s, 4, TcCtl{2000000LL, 1});
}

template void gram_tc<double>(const double*, const double*, int, int, int, double*, double*, int, int*, cudaStream_t,
                              bool);
template void gram_tc<float>(const float*, const float*, int, int, int, double*, double*, int, int*, cudaStream_t,
                             bool);
template void expand_tc<double>(const double*, const double*, const double*, int, int, int, int, double*,
                                unsigned char*, int*, cudaStream_t);
template void expand_tc<float>(const float*, const float*, const double*, int, int, int, int, float*, unsigned char*,
                               int*, cudaStream_t);

}  // namespace bmg
