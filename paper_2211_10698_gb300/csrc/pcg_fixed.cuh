// Exact sums of FP64 values in fixed point, and a device-wide barrier that carries them.
//
// The dot products of a CG iteration are summed over every thread of every block.  In FP64
// that sum is a chain of dependent additions on the narrow FP64 pipe of this part (64 pipe
// cycles per warp instruction), first inside each block and then, after the grid barrier,
// over the blocks' partials: together more than a microsecond of every iteration.  Here each
// thread turns its partial into integers instead, and the sums run on the integer units:
//
//   * A window 2^lo .. 2^(lo + kFxTop) is shared by all blocks (derived from the previous
//     iteration's sums, which every block holds identically).  A value v = +-m 2^e becomes
//     X = trunc(|v| 2^-lo) < 2^kFxTop, written as kFxDigits digits of kFxBits bits each; the
//     sign is applied to every digit, so no carry ever crosses digits.
//   * A warp adds its lanes' digits with one redux.sync per digit (|sum| < 2^31), a block its
//     warps' digit sums in 64-bit integers (|sum| < 2^35).
//   * Each block adds, per digit, (1 << kFxCountShift) + kFxBias + its digit sum to one 64-bit
//     word in global memory (one release reduction per word).  The top bits of a word count
//     the blocks that have added to it, so a word is complete when its count equals the
//     number of blocks: the wait on the words is the grid barrier, and the same load that
//     ends it delivers the sums (one L2 round trip instead of a barrier and then a load of
//     every block's partial).
//   * The digit sums are recombined in 128-bit integer arithmetic, exactly, and rounded once
//     to FP64 (to nearest, ties to even).
//
// Integer addition is associative, so the result does not depend on the order in which
// threads or blocks add: it is bitwise reproducible and more accurate than an FP64 tree (the
// only errors are the truncation of each value below 2^lo, below 2^-88 of the largest
// previous sum, and the final rounding).  A value that does not fit the window (a sum grew
// more than 2^kFxMargin-fold in one iteration, or is not finite) is counted in an extra
// word; every block then sees the count and repeats the reduction in FP64 (the fallback).
//
// Two buffers of words alternate by reduction index and are never cleared during a solve: a
// block keeps each buffer's last complete words and takes the difference, in which counts and
// digit sums both come out modulo 2^64.  A block adds to reduction i + 2 only after its wait of
// reduction i + 1, to which every block has added only after its own wait of reduction i, so no
// word of reduction i changes while a block still reads it.
//
// The words carry all that the reduction needs.  Where other data must be visible after the
// wait (vectors in global memory that other blocks read), the arrival is a release and the
// wait an acquire; where neighbours exchange their data in tagged slots (tag_put, tag_get
// below) both are relaxed, which takes the wait for the block's outstanding stores out of
// every iteration.
#pragma once
#include <cstring>

#include "pcg_common.cuh"

namespace ccm {

constexpr int kFxDigits = 5;                             // digits per value
constexpr int kFxBits = 26;                              // bits per digit
constexpr int kFxQ = 3;                                  // values per reduction
// A singular system's residual keeps clear of the null space (the constants: D^1/2 1 in the scaled system) in
// exact arithmetic only.  Rounding of K's rows adds to the null component in every iteration, nothing ever
// reduces it, and once it is as large as the residual alpha and beta are wrong: at 192x192 a tolerance of
// 1e-13 took 1735 iterations instead of 977, and a right-hand side of mean 1e6 times its variation was not
// solved at all.  So reductions 1, 1 + kZeroMeanEvery, ... go through the FP64 rows with a fourth sum, the
// residual's component, which is then taken out (a few us each: under 3 % of a small solve's time).
constexpr int kZeroMeanEvery = 64;
static_assert(kFxWords == kFxQ * kFxDigits + 1, "digit sums, then the overflow count");
constexpr int kFxCountShift = 50;                        // arrivals counted in bits 50..63
constexpr long long kFxBias = 1LL << 40;                 // keeps a block's addend positive
constexpr int kFxTop = 108;                              // |X| < 2^108: 2^18 summands stay below 2^126
constexpr int kFxMargin = 20;                            // window top: 2^20 times the largest previous sum
static_assert(kFxDigits * kFxBits >= kFxTop + 18, "digits cover the sum's range");
static_assert(kFxWords <= 32, "one lane per word");

// The arithmetic below is plain integer work on bit patterns, the same on the host (where the
// tests check it against exact rational sums) and on the device.
__host__ __device__ __forceinline__ long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}
__host__ __device__ __forceinline__ double fx_double(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, sizeof x);
  return x;
#endif
}
__host__ __device__ __forceinline__ int fx_clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x == 0 ? 64 : __builtin_clzll(x);
#endif
}

// Window bottom for values of the size of a, b, c: 2^lo with 2^(lo + kFxTop) = 2^kFxMargin
// times the largest of their powers of two.  Integer work on the bit patterns only.
__host__ __device__ __forceinline__ int fx_window(double a, double b, double c) {
  auto ex = [](double x) { return (int)((fx_bits(x) >> 52) & 0x7ff); };
  int e = ex(a), eb = ex(b), ec = ex(c);
  if (eb > e) e = eb;
  if (ec > e) e = ec;
  if (e == 0x7ff) e = 1023;  // not finite: the solve stops on it; any window will do
  if (e == 0) e = 1;         // zero or subnormal
  return (e - 1023) + kFxMargin - kFxTop;
}

// The digits of v in the window of bottom 2^lo; false if v does not fit (or is not finite),
// in which case the digits are zero.
__host__ __device__ __forceinline__ bool fx_digits(double v, int lo, int (&d)[kFxDigits]) {
  const unsigned long long b = (unsigned long long)fx_bits(v);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & 0xfffffffffffffULL;
  int e = -1074;
  if (ex != 0) {
    m |= 1ULL << 52;
    e = ex - 1075;
  }
  int s = e - lo;  // position of m's lowest bit in the window
  const bool ok = ex != 0x7ff && (m == 0 || s + 53 <= kFxTop);
  if (!ok) m = 0;
  if (s < 0) {
    m = s > -64 ? m >> -s : 0;
    s = 0;
  }
  // m (53 bits) shifted by the offset in its lowest digit covers three digits, w0 .. w0 + 2
  static_assert(kFxBits == 26 && kFxDigits == 5 && kFxTop <= 108, "three digits, the lowest of them one of 0, 1, 2");
  const int w0 = s >= 2 * kFxBits ? 2 : (s >= kFxBits ? 1 : 0), off = s - kFxBits * w0;
  constexpr unsigned int mask = (1u << kFxBits) - 1;
  int p0 = (int)((unsigned int)(m << off) & mask);
  int p1 = (int)((unsigned int)(m >> (kFxBits - off)) & mask);
  int p2 = (int)(unsigned int)((m >> (kFxBits - off)) >> kFxBits);
  if (b >> 63) {
    p0 = -p0;
    p1 = -p1;
    p2 = -p2;
  }
  d[0] = w0 == 0 ? p0 : 0;
  d[1] = w0 == 0 ? p1 : (w0 == 1 ? p0 : 0);
  d[2] = w0 == 0 ? p2 : (w0 == 1 ? p1 : p0);
  d[3] = w0 == 1 ? p2 : (w0 == 2 ? p1 : 0);
  d[4] = w0 == 2 ? p2 : 0;
  return ok;
}

// x 2^k for |k| <= 2044: two multiplications by normal powers of two (exact unless the
// result is subnormal).
__host__ __device__ __forceinline__ double fx_scale(double x, int k) {
  const int k1 = k / 2, k2 = k - k1;
  return (x * fx_double((long long)(k1 + 1023) << 52)) * fx_double((long long)(k2 + 1023) << 52);
}

// sum_k S[k] 2^(kFxBits k + lo), exactly in 128-bit integers (the true sum is below 2^126
// in magnitude), then rounded once to FP64.
__host__ __device__ __forceinline__ double fx_value(const long long* S, int lo) {
  unsigned __int128 X = 0;
#pragma unroll
  for (int k = 0; k < kFxDigits; ++k) X += (unsigned __int128)(__int128)S[k] << (kFxBits * k);
  const bool neg = (__int128)X < 0;
  const unsigned __int128 U = neg ? (unsigned __int128)0 - X : X;
  if (U == 0) return 0.0;
  const unsigned long long hi = (unsigned long long)(U >> 64), lw = (unsigned long long)U;
  const int n = hi ? 128 - fx_clz64(hi) : 64 - fx_clz64(lw);  // bit length
  // T = the significand, 53 bits, and the value T 2^(lo + sh)
  unsigned long long T;
  int sh = n - 53;
  if (sh <= 0) {
    T = lw << (-sh);  // exact
  } else {
    T = (unsigned long long)(U >> sh);
    const unsigned __int128 rem = U & (((unsigned __int128)1 << sh) - 1);
    const unsigned __int128 half = (unsigned __int128)1 << (sh - 1);
    if (rem > half || (rem == half && (T & 1))) T += 1;  // to nearest, ties to even
    if (T >> 53) {  // rounded up to 2^53
      T >>= 1;
      sh += 1;
    }
  }
  // assembled from its fields when the result is normal (integer work only), otherwise scaled
  const int E = lo + sh + 52 + 1023;  // biased exponent of T 2^(lo + sh), T in [2^52, 2^53)
  const unsigned long long sign = neg ? 1ULL << 63 : 0ULL;
  if (E >= 1 && E <= 2046)
    return fx_double((long long)(sign | ((unsigned long long)E << 52) | (T & 0xfffffffffffffULL)));
  const double r = fx_scale((double)T, lo + sh);
  return neg ? -r : r;
}

// Loads of a polled word: acquire, or relaxed where the word itself is all that is read.
template <bool ACQ>
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  if constexpr (ACQ) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  else asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// A value and its tag in one 16-byte slot, written and read as one 128-bit access: a reader
// that finds the tag it expects has the value that was stored with it, whatever else is in
// flight, so neighbours exchange values without a fence.
__device__ __forceinline__ void tag_put(ulonglong2* slot, double v, unsigned int tag) {
  const unsigned __int128 w = ((unsigned __int128)tag << 64) | (unsigned long long)__double_as_longlong(v);
  asm volatile("st.relaxed.gpu.global.b128 [%0], %1;" ::"l"(slot), "q"(w) : "memory");
}
// true with the slot's value in v if it carries `tag`
__device__ __forceinline__ bool tag_get(const ulonglong2* slot, unsigned int tag, double& v) {
  unsigned __int128 w;
  asm volatile("ld.relaxed.gpu.global.b128 %0, [%1];" : "=q"(w) : "l"(slot) : "memory");
  v = __longlong_as_double((long long)(unsigned long long)w);
  return (unsigned long long)(w >> 64) == tag;
}

// tag_get until the slot carries `tag`, within `budget` cycles (else *err is raised and false returned)
__device__ __forceinline__ bool tag_wait(const ulonglong2* slot, unsigned int tag, double& v, long long budget,
                                         int* err) {
  const long long t0 = clock64();
  while (!tag_get(slot, tag, v)) {
    if (clock64() - t0 > budget) {
      atomicExch(err, 1);
      return false;
    }
  }
  return true;
}

// Shared state of one block's fixed-point reduction: per-warp digit sums of NT threads.
template <int NT>
struct FxShared {
  int w[NT / 32][kFxWords];
};

// The digits of v[0..2] summed per warp into sh (each of the NT threads).
template <int NT>
__device__ __forceinline__ void fx_block_digits(const double (&v)[4], int lo, FxShared<NT>& sh) {
  int d[kFxWords];
  bool fit = true;
#pragma unroll
  for (int q = 0; q < kFxQ; ++q) {
    int dq[kFxDigits];
    fit = fx_digits(v[q], lo, dq) && fit;
#pragma unroll
    for (int k = 0; k < kFxDigits; ++k) d[q * kFxDigits + k] = dq[k];
  }
  d[kFxWords - 1] = fit ? 0 : 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kFxWords; ++k) d[k] = __reduce_add_sync(0xffffffffu, d[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < kFxWords; ++k) sh.w[wid][k] = d[k];
}

// Arrival, by one whole warp after every warp's digits are in sh: the block's digit sums added
// to the words of buffer `buf`.  REL: what the warp has seen (its barrier with the others
// included) is released with the words.
template <int NT, bool REL>
__device__ __forceinline__ void fx_arrive(unsigned long long* acc, int buf, bool absent, const FxShared<NT>& sh) {
  const int lane = threadIdx.x & 31;
  if (lane < kFxWords) {
    long long s = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) s += sh.w[w][lane];
    const unsigned long long word = (1ULL << kFxCountShift) + (unsigned long long)(s + kFxBias);
    unsigned long long* dst = acc + ((size_t)buf * kFxWords + lane) * kFxStride;
    if (!absent) {
      if constexpr (REL) asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(dst), "l"(word) : "memory");
      else asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst), "l"(word) : "memory");
    }
  }
}

// Wait, by one whole warp: until all nb blocks have added to every word of buffer `buf`
// (bounded by `budget` cycles; on give-up *err is raised and false returned).  last: this lane's
// word of that buffer after its previous use (0 at first), updated.  digit: the grid's sum of
// this lane's word (lanes below kFxWords).
template <bool ACQ>
__device__ __forceinline__ bool fx_wait(const unsigned long long* acc, int buf, int nb, long long budget, int* err,
                                        unsigned long long& last, long long& digit) {
  const int lane = threadIdx.x & 31;
  const unsigned long long* src = acc + ((size_t)buf * kFxWords + (lane < kFxWords ? lane : 0)) * kFxStride;
  unsigned long long w = 0, d = 0;
  const long long t0 = clock64();
  while (true) {
    w = ld_word<ACQ>(src);
    d = w - last;
    if (__all_sync(0xffffffffu, (d >> kFxCountShift) == (unsigned long long)nb)) break;
    if (__shfl_sync(0xffffffffu, clock64() - t0 > budget ? 1 : 0, 0)) {
      if (lane == 0) atomicExch(err, 1);
      return false;
    }
  }
  last = w;
  digit = (long long)(d & ((1ULL << kFxCountShift) - 1)) - (long long)nb * kFxBias;
  return true;
}

}  // namespace ccm
