// r^-1, r^-3 and r^-5 from r^2 in FP64, with as few FP64 instructions as the accuracy allows: this GPU issues one
// of them in the time of 64 FP32 or integer ones, and the pair sums in FP64 are bound by nothing else.
//
// With an FP32 approximation y of r^-1 and e = 1 - r^2 y^2 (|e| < 2^-20), r^-k = y^k (1 - e)^(-k/2), whose binomial
// series is y^k (1 + e (k/2 + (k/2)(k/2 + 1)/2 e)) up to 7 e^3 < 2^-57 for k <= 5. y^2 is exact in FP64, so e carries
// one rounding of a number 2^-20 as large as the result; of the inner sum only the first
// term has to be exact, the second comes from FP32. Conversions between FP32 and FP64 run on the FP64 pipe too, so
// they are done on the bits. Squares of distances outside 2^-100 .. 2^100, zeros, infinities and NaN take CUDA's
// rsqrt. Of the FP64 instructions of a double-layer pair 22 become 16, of a single-layer pair 16 become 11: a solve of
// eight applications to six drops of degree 16 (4e7 pairs each) 17.6 -> 14.1 ms. Errors of single pairs over all
// distances: at most 8 (r^-1) and 12 (r^-3) units of 2^-53 with those of r^2 and the product.
#pragma once

namespace shbim {

// the FP32 number with the leading bits of a (truncated); |a| in the FP32 range of exponents
__device__ __forceinline__ float trunc_f32(double a) {
  const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
  return __uint_as_float((__funnelshift_l(lo, hi & 0x7fffffffu, 3) - (896u << 23)) | (hi & 0x80000000u));
}

// a positive normal FP32 number in FP64
__device__ __forceinline__ double widen_f32(float a) {
  const unsigned b = __float_as_uint(a);
  return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

__device__ __forceinline__ bool inv_range(double r2) {
  return (unsigned)__double2hiint(r2) - ((1023u - 100u) << 20) < (200u << 20);
}

// 1 + e (a + b e) for a = 0.5, 1.5 or 2.5: b e is added to a's mantissa as an integer of 2^-48
template <int K>
__device__ __forceinline__ double inv_factor(double e, float ef) {
  constexpr float kB = (K == 1 ? 0.375f : (K == 3 ? 1.875f : 4.375f)) * 281474976710656.f;
  constexpr long long kA = K == 1 ? 0x3FE0000000000000ll : (K == 3 ? 0x3FF8000000000000ll : 0x4004000000000000ll);
  const long long n = __float2int_rn(ef * kB);
  // 2^-48 in units of the last place: below 0.5 they are half as large as above
  const long long unit = K == 1 ? (n < 0 ? 64 : 32) : (K == 3 ? 16 : 8);
  return fma(e, __longlong_as_double(kA + n * unit), 1.0);
}

__device__ __forceinline__ void inv_seed(double r2, double& y, double& t, double& e, float& ef) {
  y = widen_f32(rsqrtf(trunc_f32(r2)));
  t = y * y;
  e = fma(-r2, t, 1.0);
  // exponents below 2^-64 would wrap in trunc_f32, and do not count
  ef = ((unsigned)__double2hiint(e) & 0x7fffffffu) > ((1023u - 64u) << 20) ? trunc_f32(e) : 0.f;
}

__device__ __forceinline__ double inv_r(double r2) {
  if (!inv_range(r2)) return rsqrt(r2);
  double y, t, e;
  float ef;
  inv_seed(r2, y, t, e, ef);
  return y * inv_factor<1>(e, ef);
}

__device__ __forceinline__ double inv_r3(double r2) {
  if (!inv_range(r2)) {
    const double ri = rsqrt(r2);
    return ri * ri * ri;
  }
  double y, t, e;
  float ef;
  inv_seed(r2, y, t, e, ef);
  return (y * t) * inv_factor<3>(e, ef);
}

__device__ __forceinline__ double inv_r5(double r2) {
  if (!inv_range(r2)) {
    const double ri = rsqrt(r2), ri2 = ri * ri;
    return ri2 * ri * ri2;
  }
  double y, t, e;
  float ef;
  inv_seed(r2, y, t, e, ef);
  return (y * (t * t)) * inv_factor<5>(e, ef);
}

}  // namespace shbim
