// Scalars and warp sums of the Householder kernels (k_qr_smem.cu,
// k_qr_blocked.cu), arranged for few FP64 instructions: one of them occupies
// its SM quarter for 64 to 76 clocks.
#pragma once

#include "common.cuh"

namespace dqmc {

// x 2^e for a normal x and a normal result, in the exponent field.
__device__ __forceinline__ double qs_scale2(double x, int e) {
  return __longlong_as_double(__double_as_longlong(x) + (static_cast<long long>(e) << 52));
}

// Squared norms from 2^1020 on (this high word): sums that the reflector needs,
// up to twice the largest squared norm, could leave the range of FP64, and the
// reciprocal its normal numbers, although the columns do neither.  The columns
// are then scaled by kQsDown before the first step and R by kQsUp after the
// last; no further down, as the smallest columns of such a product lie near the
// lower end of the range.
constexpr unsigned kQsBig = 2043u << 20, kQsNonFinite = 0x7FF00000u;
constexpr double kQsDown = 0x1p-4, kQsUp = 0x1p4;

// The leading 24 bits of a double in [1, 4) as a float, and a float as a
// double, in integer arithmetic (a conversion would take the FP64 pipe).
__device__ __forceinline__ float qs_to_f(double x) {
  return __int_as_float(static_cast<int>((__double_as_longlong(x) >> 29) - (896LL << 23)));
}
__device__ __forceinline__ double qs_to_d(float x) {
  return __longlong_as_double((static_cast<long long>(__float_as_int(x)) << 29) + (896LL << 52));
}

// Scalars of the reflector of (alpha, x), sigma = |x|^2 (see above): beta,
// vj = v[j] and kap = 1 / (s u) = 1 / (n2 + |alpha| s), n2 = alpha^2 + sigma.
// The square root and the reciprocal start from the FP32 approximations and
// take one third-order Householder iteration each (relative error e of the
// start, e^3 of the result): ten dependent FP64 instructions instead of the
// thirty of sqrt() and a division.
__device__ __forceinline__ void qs_reflector(double alpha, double sigma, double& beta, double& kap,
                                             double& vj) {
  beta = alpha;
  kap = 0.0;
  vj = 0.0;
  if (__double_as_longlong(sigma) == 0LL) return;
  const double n2 = fma(alpha, alpha, sigma), aa = absd(alpha);
  const int E = static_cast<int>((__double_as_longlong(n2) >> 52) & 0x7FF);
  double s;
  if (E > 8 && E < 2036) {
    const int e = (E - 1023) & ~1;            // n2 = m 2^e, m in [1, 4)
    const double m = qs_scale2(n2, -e);
    const double y0 = qs_to_d(rsqrtf(qs_to_f(m)));
    const double t = m * y0;                  // about sqrt(m)
    const double e1 = fma(-t, y0, 1.0);
    const double q = e1 * fma(e1, 0.375, 0.5);
    s = qs_scale2(fma(t, q, t), e / 2);
    const double su = fma(aa, s, n2);         // in [n2, 2 n2]
    const int eu = static_cast<int>((__double_as_longlong(su) >> 52) & 0x7FF) - 1023;
    const double mu = qs_scale2(su, -eu);
    const double r0 = qs_to_d(__fdividef(1.0f, qs_to_f(mu)));
    const double e2 = fma(-mu, r0, 1.0);
    kap = qs_scale2(fma(r0, fma(e2, e2, e2), r0), -eu);
  } else {  // squares near the ends of the range (or not finite)
    s = sqrt(n2);
    kap = 1.0 / fma(aa, s, n2);
  }
  // comparisons on the sign bit (an FP64 one would take the FP64 pipe)
  beta = (__double_as_longlong(alpha) < 0) ? s : -s;
  vj = alpha - beta;
}

// Warp sum of non-negative finite numbers in 64-bit fixed point: aligned to
// the largest exponent (58 bits, rounded), three integer warp reductions
// instead of five rounds of shuffles and FP64 additions (about 130 against 650
// clocks).  Error below 2^-52 of the sum: up to 15.5 units of 2^-57 of the
// largest term's power of two, and the rounding of the sum.  Non-finite input
// gives non-finite output.
__device__ __forceinline__ double qs_warp_sum_pos(double a) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(a));
  const int E = static_cast<int>((bits >> 52) & 0x7FF);
  const int Emax = static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, static_cast<unsigned>(E)));
  if (Emax == 0x7FF) return __longlong_as_double(0x7FF8000000000000LL);
  unsigned long long f = 0ull;
  const int sh = Emax - E;
  if (E != 0 && sh < 59) {
    f = ((bits & ((1ull << 52) - 1)) | (1ull << 52)) << 5;
    f = (f + ((1ull << sh) >> 1)) >> sh;
  }
  const unsigned l0 = static_cast<unsigned>(f) & 0x3FFFFFu, l1 = static_cast<unsigned>(f >> 22) & 0x3FFFFFu,
                 l2 = static_cast<unsigned>(f >> 44);
  const unsigned long long s = static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l0)) +
                               (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l1)) << 22) +
                               (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l2)) << 44);
  if (s == 0ull) return 0.0;
  // s 2^(Emax - 1023 - 57); s in [2^57, 2^63)
  const double d = __ull2double_rn(s);
  const int e = Emax - 1023 - 57;
  if (Emax > 64 && Emax < 2040) return __longlong_as_double(__double_as_longlong(d) + (static_cast<long long>(e) << 52));
  return ldexp(d, e);
}

// The same for numbers of either sign: a bias of 2^58 per lane keeps the words
// non-negative.  Error below 2^-53 of the largest term, and the rounding of the
// sum.
__device__ __forceinline__ double qs_warp_sum(double a) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(a));
  const int E = static_cast<int>((bits >> 52) & 0x7FF);
  const int Emax = static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, static_cast<unsigned>(E)));
  if (Emax == 0x7FF) return __longlong_as_double(0x7FF8000000000000LL);
  unsigned long long f = 1ull << 58;
  const int sh = Emax - E;
  if (E != 0 && sh < 59) {
    unsigned long long g = ((bits & ((1ull << 52) - 1)) | (1ull << 52)) << 5;
    g = (g + ((1ull << sh) >> 1)) >> sh;
    f = (static_cast<long long>(bits) < 0) ? f - g : f + g;
  }
  const unsigned l0 = static_cast<unsigned>(f) & 0x3FFFFFu, l1 = static_cast<unsigned>(f >> 22) & 0x3FFFFFu,
                 l2 = static_cast<unsigned>(f >> 44);
  const unsigned long long s = static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l0)) +
                               (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l1)) << 22) +
                               (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, l2)) << 44);
  const long long t = static_cast<long long>(s ^ (1ull << 63));  // s - 2^63
  if (t == 0) return 0.0;
  const double d = __ll2double_rn(t);
  const int e = Emax - 1023 - 57;
  if (Emax > 64 && Emax < 2040) return __longlong_as_double(__double_as_longlong(d) + (static_cast<long long>(e) << 52));
  return ldexp(d, e);
}

// log2 of the squared norm of x[0 .. len) as an FP32 sort key, from the
// exponent fields and the FP32 mantissas (the order only steers the
// numerics; any order gives an exact factorisation).  One warp, len <= kMaxN;
// every element is loaded once, all loads of a lane in flight together.  The
// key is returned on every lane: +3e38 for Inf/NaN entries, -3e38 for a zero
// vector.
__device__ __forceinline__ float qb_norm_key(const double* x, int len, int lane) {
  constexpr int kR = kMaxN / 32;
  long long bits[kR];
#pragma unroll
  for (int t = 0; t < kR; ++t) {
    const int r = lane + 32 * t;
    bits[t] = (r < len) ? __double_as_longlong(x[r]) : 0LL;
  }
  int emax = 0;
  bool bad = false;
#pragma unroll
  for (int t = 0; t < kR; ++t) {
    const int E = static_cast<int>((bits[t] >> 52) & 0x7FF);
    bad |= (E == 0x7FF);
    emax = max(emax, E);
  }
  for (int o = 16; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xFFFFFFFFu, emax, o));
  bad = __any_sync(0xFFFFFFFFu, bad);
  float s = 0.0f;
#pragma unroll
  for (int t = 0; t < kR; ++t) {
    const int E = static_cast<int>((bits[t] >> 52) & 0x7FF);
    if (E != 0) {
      const float mt = __int_as_float(0x3F800000 | static_cast<int>((bits[t] >> 29) & 0x7FFFFF));
      const float y = ldexpf(mt, E - emax);
      s = fmaf(y, y, s);
    }
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (bad) return 3.0e38f;
  if (emax == 0) return -3.0e38f;
  return 2.0f * static_cast<float>(emax - 1023) + __log2f(s);
}

}  // namespace dqmc
