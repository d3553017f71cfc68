// The CG scalars alpha and beta from the iteration's exact sums, in integer arithmetic.
//
// Between the arrival of the last block's digits and the next iteration every block forms the
// same two scalars: a chain of eleven dependent FP64 operations (two of them conversions), each
// of which waits its turn on an FP64 pipe that takes one warp instruction per 64 cycles and is
// busy with the vector updates of the other warps.  The integer units are idle then.  A scalar
// here is sign, 64-bit significand and exponent, so products and the reciprocal are a few
// 64-bit multiplications; every operation is correct to about 2^-61, eight bits more than FP64,
// and only alpha and beta themselves are rounded to FP64.
#pragma once
#include <cmath>

#include "pcg_fixed.cuh"

namespace ccm {

// (neg ? -1 : 1) m 2^e, m in [2^63, 2^64), or m = 0.
struct Scalar {
  unsigned long long m;
  int e;
  bool neg;
};

__host__ __device__ __forceinline__ unsigned long long sc_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}

// The leading 64 bits of a 128-bit magnitude times 2^lo.
__host__ __device__ __forceinline__ Scalar sc_of_u128(unsigned long long hi, unsigned long long lw, int lo, bool neg) {
  if (hi == 0) {
    if (lw == 0) return Scalar{0ULL, 0, false};
    const int z = fx_clz64(lw);
    return Scalar{lw << z, lo - z, neg};
  }
  const int z = fx_clz64(hi);
  return Scalar{z == 0 ? hi : (hi << z) | (lw >> (64 - z)), lo + 64 - z, neg};
}

// sum_k S[k] 2^(kFxBits k + lo) (see fx_value), its leading 64 bits.
__host__ __device__ __forceinline__ Scalar sc_of_digits(const long long* S, int lo) {
  unsigned __int128 X = 0;
#pragma unroll
  for (int k = 0; k < kFxDigits; ++k) X += (unsigned __int128)(__int128)S[k] << (kFxBits * k);
  const bool neg = (__int128)X < 0;
  if (neg) X = (unsigned __int128)0 - X;
  return sc_of_u128((unsigned long long)(X >> 64), (unsigned long long)X, lo, neg);
}

// A finite FP64 value.
__host__ __device__ __forceinline__ Scalar sc_of_double(double x) {
  const unsigned long long b = (unsigned long long)fx_bits(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & 0xfffffffffffffULL;
  if (ex != 0) m |= 1ULL << 52;
  return sc_of_u128(0ULL, m, ex != 0 ? ex - 1075 : -1074, (b >> 63) != 0);
}

// Rounded to nearest (ties to even) FP64, subnormals included; beyond its range infinite.
__host__ __device__ __forceinline__ double sc_double(const Scalar& a) {
  const unsigned long long sign = a.neg ? 1ULL << 63 : 0ULL;
  if (a.m == 0) return fx_double((long long)sign);
  int E = a.e + 63 + 1023;
  if (E < 1) {
    // subnormal: fewer bits are kept (a residual norm near the end of a solve with tiny right-hand side;
    // flushed to 0 it would meet any tolerance)
    const int shift = 12 - E;
    if (shift > 64) return fx_double((long long)sign);
    const unsigned long long half = 1ULL << (shift - 1);
    const unsigned long long rest = shift == 64 ? a.m : a.m & ((half << 1) - 1);
    unsigned long long t = shift == 64 ? 0ULL : a.m >> shift;
    if (rest > half || (rest == half && (t & 1))) t += 1;  // (2^52 is the smallest normal number)
    return fx_double((long long)(sign | t));
  }
  unsigned long long t = a.m >> 11;
  const unsigned long long rem = a.m & 0x7ffULL;
  if (rem > 0x400ULL || (rem == 0x400ULL && (t & 1))) t += 1;
  if (t >> 53) { t >>= 1; E += 1; }
  if (E > 2046) return fx_double((long long)(sign | (0x7ffULL << 52)));
  return fx_double((long long)(sign | ((unsigned long long)E << 52) | (t & 0xfffffffffffffULL)));
}

// m 2^e to nearest FP64 (m normalised, ties away from zero; the exponent field absorbs the carry of
// the rounding).
__host__ __device__ __forceinline__ double sc_double_pos(unsigned long long m, int e) {
  const int E = e + 63 + 1023;
  if (E < 1 || E > 2045) return sc_double(Scalar{m, e, false});
  return fx_double((long long)(((unsigned long long)(E - 1) << 52) + (m >> 11) + ((m >> 10) & 1ULL)));
}

__host__ __device__ __forceinline__ Scalar sc_mul(const Scalar& a, const Scalar& b) {
  if (a.m == 0 || b.m == 0) return Scalar{0ULL, 0, false};
  const unsigned long long hi = sc_mulhi(a.m, b.m), lw = a.m * b.m;
  const bool top = (hi >> 63) != 0;
  return Scalar{top ? hi : (hi << 1) | (lw >> 63), a.e + b.e + (top ? 64 : 63), a.neg != b.neg};
}

__host__ __device__ __forceinline__ Scalar sc_add(const Scalar& x, const Scalar& y) {
  if (x.m == 0) return y;
  if (y.m == 0) return x;
  const bool swap = y.e > x.e || (y.e == x.e && y.m > x.m);
  const Scalar a = swap ? y : x, b = swap ? x : y;  // |a| >= |b|
  const int d = a.e - b.e;
  const unsigned long long bm = d < 64 ? b.m >> d : 0ULL;
  if (a.neg == b.neg) {
    const unsigned long long s = a.m + bm;
    if (s < bm) return Scalar{(s >> 1) | (1ULL << 63), a.e + 1, a.neg};
    return Scalar{s, a.e, a.neg};
  }
  // one more bit of b kept, so that a difference of nearly equal values loses none
  const unsigned long long lowbit = d >= 1 && d <= 64 ? (b.m >> (d - 1)) & 1ULL : 0ULL;
  unsigned long long s = a.m - bm;
  if (lowbit) {
    // s - 1/2: as 2 s - 1 where it fits below 2^64, else truncated
    if (s >> 63) s -= 1;
    else {
      s = 2 * s - 1;
      const int z = fx_clz64(s);
      return Scalar{s << z, a.e - 1 - z, a.neg};
    }
  }
  if (s == 0) return Scalar{0ULL, 0, false};
  const int z = fx_clz64(s);
  return Scalar{s << z, a.e - z, a.neg};
}
__host__ __device__ __forceinline__ Scalar sc_neg(const Scalar& a) { return Scalar{a.m, a.e, a.m != 0 && !a.neg}; }

// 1 / a (0 for 0): with d = m / 2^64 in [1/2, 1) and X = 2^62 / d, two Newton steps
// X += X (1 - d X) from the single-precision reciprocal (2^-22, 2^-44, then about 2^-61).
__host__ __device__ __forceinline__ Scalar sc_recip(const Scalar& a) {
  if (a.m == 0) return a;
  const float f = (float)(unsigned int)(a.m >> 40);  // 2^24 d truncated, exact
  const float r = 16777216.0f / f;                   // (1, 2]
  long long X = (long long)(r * 4194304.0f) << 40;   // r 2^62
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (X < 0) X = 0x7fffffffffffffffLL;
    const long long E = (1LL << 62) - (long long)sc_mulhi(a.m, (unsigned long long)X);
    // X E 2^-62, signed
    const bool neg = E < 0;
    const unsigned long long c = sc_mulhi((unsigned long long)X, (unsigned long long)(neg ? -E : E) << 2);
    X = neg ? X - (long long)c : X + (long long)c;
  }
  const unsigned long long u = (unsigned long long)X;
  const int z = fx_clz64(u);
  // 1 / (m 2^e) = (X / 2^62) 2^(-64 - e)
  return Scalar{u << z, -126 - a.e - z, a.neg};
}

// Floor of log2 |a| (a large negative value for 0).
__host__ __device__ __forceinline__ int sc_log2(const Scalar& a) { return a.m == 0 ? -1023 : a.e + 63; }

// The recurrence's state between iterations: 1 / gamma, whose significand lies in
// [2^62, 2^63], and den with alpha = gamma / den.
struct CgState {
  Scalar igamma, den;
};

// 1 / gamma for CgState (gamma > 0).
__host__ __device__ __forceinline__ Scalar cg_inverse(const Scalar& gamma) {
  Scalar r = sc_recip(gamma);
  r.m >>= 1;
  r.e += 1;
  return r;
}

__host__ __device__ __forceinline__ float sc_rcp_approx(float x) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, x);
#else
  return 1.0f / x;
#endif
}

// a / b for normalised significands a and b (in [2^63, 2^64)): q with q / 2^62 close to
// a / b, q in (2^61, 2^63): the single-precision reciprocal of b (about 2^-22), then two
// corrections of the quotient by its remainder (2^-44, then a few units of 2^-61).
__host__ __device__ __forceinline__ unsigned long long sc_quotient(unsigned long long a, unsigned long long b) {
  const float f = (float)(unsigned int)(b >> 40);  // 2^24 b / 2^64 truncated, exact
  // X 2^-30 is about 2^64 / b, in (1, 2]; kept below 2^31
  const unsigned int X = (unsigned int)fminf(sc_rcp_approx(f) * 18014398509481984.0f, 2147483520.0f);
  unsigned long long q = sc_mulhi(a, (unsigned long long)X << 32);  // a / b 2^62
  long long r = (long long)(a >> 2) - (long long)sc_mulhi(q, b);     // |r| < 2^42
#ifdef __CUDA_ARCH__
  q += (unsigned long long)(__mul64hi(r << 18, (long long)((unsigned long long)X << 32)) >> 16);
#else
  q += (unsigned long long)(((__int128)r * X) >> 30);
#endif
  r = (long long)(a >> 2) - (long long)sc_mulhi(q, b);               // |r| < 2^20
  q += (unsigned long long)((r * (long long)X) >> 30);
  return q;
}

#ifdef __CUDACC__
// The grid's three sums in s[0..2] of lane 0, and in every lane its count of values outside the
// window in *overflow, from a warp whose lanes hold the digit sums (fx_wait).
__device__ __forceinline__ void fx_sums(long long digit, int lo, Scalar (&s)[3], int* overflow) {
  *overflow = (int)__shfl_sync(0xffffffffu, digit, kFxWords - 1);
  // lane q assembles quantity q (the other lanes repeat quantity lane % 3)
  long long S[kFxDigits];
  const int q = (threadIdx.x & 31) % kFxQ;
#pragma unroll
  for (int k = 0; k < kFxDigits; ++k) S[k] = __shfl_sync(0xffffffffu, digit, q * kFxDigits + k);
  s[0] = sc_of_digits(S, lo);
  const int en = 2 * s[0].e + (s[0].neg ? 1 : 0);
#pragma unroll
  for (int k = 1; k < kFxQ; ++k) {
    s[k].m = __shfl_down_sync(0xffffffffu, s[0].m, k);
    const int e = __shfl_down_sync(0xffffffffu, en, k);
    s[k].e = e >> 1;
    s[k].neg = (e & 1) != 0;
  }
}
#endif

// Chronopoulos-Gear: beta = gamma / gamma_old, den = delta - beta gamma / alpha_old with
// 1 / alpha_old = den_old / gamma_old, alpha = gamma / den (unchanged when den = 0).
__host__ __device__ __forceinline__ void cg_scalars(const Scalar& gamma, const Scalar& delta, CgState& st, double& alpha,
                                                    double& beta) {
  // beta and beta^2 den_old, products left unnormalised (57 bits or more)
  const unsigned long long b = sc_mulhi(gamma.m, st.igamma.m);
  const int eb = gamma.e + st.igamma.e + 64;
  const unsigned long long t = sc_mulhi(sc_mulhi(b, b), st.den.m);
  const int et = 2 * eb + st.den.e + 128;
  const int d = et - delta.e;
  const bool usual = !gamma.neg && gamma.m != 0 && !delta.neg && delta.m != 0 && st.igamma.m != 0 && !st.den.neg &&
                     (d <= 0 || (d < 64 && t < (delta.m >> d)));
  if (usual) {
    const unsigned long long ta = d <= 0 ? (d > -64 ? t >> -d : 0ULL) : t << d;
    const unsigned long long r = delta.m - ta;
    if (r != 0) {
      const int z = fx_clz64(r);
      st.den = Scalar{r << z, delta.e - z, false};
      const unsigned long long q = sc_quotient(gamma.m, st.den.m);
      const int zq = fx_clz64(q);
      alpha = sc_double_pos(q << zq, gamma.e - st.den.e - 62 - zq);
      const int zb = fx_clz64(b);
      beta = sc_double_pos(b << zb, eb - zb);
      return;
    }
  }
  // a sum that is zero or negative (the recurrence has broken down)
  const Scalar bn = sc_mul(gamma, sc_of_u128(0ULL, st.igamma.m, st.igamma.e, st.igamma.neg));
  st.den = sc_add(delta, sc_neg(sc_mul(sc_mul(bn, bn), st.den)));
  beta = sc_double(bn);
  if (st.den.m != 0) alpha = sc_double(sc_mul(gamma, sc_recip(st.den)));
}

}  // namespace ccm
