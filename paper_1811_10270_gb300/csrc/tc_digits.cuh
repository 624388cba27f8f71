// The digit arithmetic of the tensor-core kernels with FP64-class accuracy (tc.cuh), kept apart
// from the PTX so that the CPU tests can compile it with a host compiler (as the double-float
// header): digit splitting of FP64 table values on the host, of double-float values in the kernels,
// and the recombination of the six exact FP32 diagonal sums. Host builds must not contract or
// reassociate floating-point operations (-ffp-contract=off).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "dfloat.cuh"

#ifdef __CUDACC__
#define TC_FN __host__ __device__ __forceinline__
#else
#define TC_FN inline
#endif

namespace shbim {
namespace tc {

constexpr int kDig = 6;          // digits per value (42 bits)
constexpr int kDig7 = 7;         // the same with one more digit (49 bits: all of a double-float value)

// digits of x 2^(42 - e), |x| < 2^e: d_0..d_4 balanced base 2^7, d_5 the rest (host)
inline void digits_host(double x, int e, int d[kDig]) {
  long long X = std::llrint(std::ldexp(x, 42 - e));
  for (int j = 0; j < kDig - 1; ++j) {
    const long long dj = ((X + 64) & 127) - 64;
    d[j] = (int)dj;
    X = (X - dj) / 128;
  }
  d[kDig - 1] = (int)X;
}

// digits of x 2^(42 - e) (ND = 6) or x 2^(49 - e) (ND = 7), |x| < 2^e: balanced base 2^7, the top one the rest (host)
inline void digits_host_n(double x, int e, int nd, int* d) {
  long long X = std::llrint(std::ldexp(x, 7 * nd - e));
  for (int j = 0; j < nd - 1; ++j) {
    const long long dj = ((X + 64) & 127) - 64;
    d[j] = (int)dj;
    X = (X - dj) / 128;
  }
  d[nd - 1] = (int)X;
}

// bfloat16 bits of a small integer (|v| <= 256 is exact: the low 16 bits of the float are zero)
inline uint16_t bf16_int(int v) {
  const float f = (float)v;
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return (uint16_t)(u >> 16);
}

// nearest integer (ties to even) of |t| < 2^22 by adding and taking away 1.5 2^23: two additions on the FP32 pipe, where
// rintf is one instruction of a pipe an eighth as wide
TC_FN float rint_fast(float t) { return dfl::sub_rn(dfl::add_rn(t, 12582912.f), 12582912.f); }

// Six balanced base-2^7 digits of y = yh + yl (|yh| < 128, |yl| <= ulp(yh) / 2), top first:
// d5 = rint(y), then the digits of the remainder times 128, and so on. The top three come from yh
// alone (every remainder exact); yl joins through one two-sum at the scale of d2; the last two come
// from an FP32 remainder whose rounding (< 2^-25 of d2's unit) stays far below d0's half unit.
// Bounds: |d5| <= 128, |d4|, |d3| <= 64, |d2| <= 72, |d1|, |d0| <= 65.
TC_FN void digits6(float yh, float yl, float (&d)[kDig]) {
  float t = yh;
  d[5] = rint_fast(t);
  t = (t - d[5]) * 128.f;
  d[4] = rint_fast(t);
  t = (t - d[4]) * 128.f;
  d[3] = rint_fast(t);
  t = (t - d[3]) * 128.f;
  const dfl::df u = dfl::two_sum(t, yl * 2097152.f);   // yl at the scale of d2 (2^21)
  d[2] = rint_fast(u.hi);
  float r = ((u.hi - d[2]) + u.lo) * 128.f;
  d[1] = rint_fast(r);
  r = (r - d[1]) * 128.f;
  d[0] = rint_fast(r);
}

// The same with ND digits, d[ND - 1] the top one: ND = 7 takes one more from the remainder, whose rounding (2^-26 of
// the unit of the fourth digit) lies below the seventh digit's half unit.
template <int ND>
TC_FN void digits_n(float yh, float yl, float (&d)[ND]) {
  float t = yh;
  d[ND - 1] = rint_fast(t);
  t = (t - d[ND - 1]) * 128.f;
  d[ND - 2] = rint_fast(t);
  t = (t - d[ND - 2]) * 128.f;
  d[ND - 3] = rint_fast(t);
  t = (t - d[ND - 3]) * 128.f;
  const dfl::df u = dfl::two_sum(t, yl * 2097152.f);
  d[ND - 4] = rint_fast(u.hi);
  float r = ((u.hi - d[ND - 4]) + u.lo) * 128.f;
  for (int j = ND - 5; j > 0; --j) {
    d[j] = rint_fast(r);
    r = (r - d[j]) * 128.f;
  }
  d[0] = rint_fast(r);
}

// Largest |digit| by position (row operand after digits6; table operand after digits_host) and the
// worst case of diagonal sum s (products with j_a + j_b = s + 5) over K products: every tensor-core
// kernel asserts at compile time that this stays below 2^24 at its longest K, so that the FP32
// accumulation in tensor memory is exact.
constexpr int kRowDigitMax[kDig] = {65, 65, 72, 64, 64, 128};
constexpr int kTabDigitMax[kDig] = {64, 64, 64, 64, 64, 128};
constexpr long long diag_sum_bound(int K, int s) {
  long long w = 0;
  for (int ja = 0; ja < kDig; ++ja) {
    const int jb = s + kDig - 1 - ja;
    if (jb >= 0 && jb < kDig) w += (long long)kRowDigitMax[ja] * kTabDigitMax[jb];
  }
  return w * K;
}
constexpr bool diag_sums_exact(int K) {
  for (int s = 0; s < kDig; ++s)
    if (diag_sum_bound(K, s) >= (1LL << 24)) return false;
  return true;
}

// The same bound for seven digits (digits_n<7>, digits_host_n): row digits at most 65 (the lowest three), 72, 64, 64
// and 128, table digits 64 and 128 at the top.
constexpr int kRowDigitMax7[kDig7] = {65, 65, 65, 72, 64, 64, 128};
constexpr int kTabDigitMax7[kDig7] = {64, 64, 64, 64, 64, 64, 128};
constexpr bool diag_sums_exact7(int K) {
  for (int s = 0; s < kDig7; ++s) {
    long long w = 0;
    for (int ja = 0; ja < kDig7; ++ja) {
      const int jb = s + kDig7 - 1 - ja;
      if (jb >= 0 && jb < kDig7) w += (long long)kRowDigitMax7[ja] * kTabDigitMax7[jb];
    }
    if (w * K >= (1LL << 24)) return false;
  }
  return true;
}

// sum_s acc_s 2^(7 (s - ND + 1)) as a double-float from the ND exact FP32 diagonal sums, acc[ND - 1] the top one:
// the leading ones joined by two-sums, the three lowest in plain FP32 as below
template <int ND>
TC_FN dfl::df combine_n(const float (&a)[ND]) {
  float low = a[0];
  low = fmaf(low, 0x1p-7f, a[1]);
  low = fmaf(low, 0x1p-7f, a[2]);
  float w = 0x1p-7f;
  dfl::df s{a[ND - 1], 0.f};
  float e = 0.f;
  for (int k = ND - 2; k > 2; --k) {
    const dfl::df t = dfl::two_sum(s.hi, a[k] * w);
    s.hi = t.hi;
    e += t.lo;
    w *= 0x1p-7f;
  }
  return dfl::quick_two_sum(s.hi, fmaf(low, w, e));
}

// sum_s acc_s 2^(7 (s - 5)) as a double-float from the six exact FP32 diagonal sums
// (|acc_s| < 2^24): the three top terms are exact in FP32 and joined by two-sums; the three lowest
// (weights 2^-21 and below) are summed in plain FP32, rounding below 2^-21 units of the top term.
TC_FN dfl::df combine6(float a5, float a4, float a3, float a2, float a1, float a0) {
  const float low = fmaf(a0, 0x1p-35f, fmaf(a1, 0x1p-28f, a2 * 0x1p-21f));
  const dfl::df s1 = dfl::two_sum(a5, a4 * 0x1p-7f);
  const dfl::df s2 = dfl::two_sum(s1.hi, a3 * 0x1p-14f);
  return dfl::quick_two_sum(s2.hi, (s1.lo + s2.lo) + low);
}

}  // namespace tc
}  // namespace shbim
