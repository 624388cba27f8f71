// Sums between well-separated drops through multipole and local expansions (Greengard and Rokhlin's
// fast multipole method with the drops as its clusters): the same regular rule (Eq. reg_quadrature) as
// the direct sums of pairs.cu, to a truncation error below the arithmetic's own.
//
// Each drop's sources act on the targets of a far drop through harmonic potentials Phi = sum q / r of
// point charges (or dipoles): one for the Laplace kernels, four for the Stokes kernels,
//   S_i   = phi_i - x_k d_i phi_k + d_i psi,           phi_k from charges f_k, psi from y.f
//   D_i   = (Phi_i - x_k d_i Phi_k + d_i Psi) / 6       for d (d.u)(d.n) / r^5, with dipole moments
//           u_k n + n_k u (Phi_k) and (y.u) n + (y.n) u (Psi)
// (positions relative to the target drop's centre; psi is shifted with it). Per application
//   1. k_far_charges, k_far_p2m, k_far_vsum, k_far_dipoles: moments of every drop about its centre;
//   2. k_far_m2l: per (far pair, potential) the moments are rotated so that the pair's axis is z (Dz Dq^T Dz Dq,
//      Dq the fixed matrix of Rx(pi/2)), translated along it order by order, rotated back;
//   3. k_far_lsum, k_far_lset: a drop's local expansion (sum over its far drops in a fixed order) and the
//      expansions of the derivatives its targets need;
//   4. k_far_l2p: values at the targets, added to the operator values;
//   5. k_far_mset, k_far_m2p, k_far_msum: drops too close for this, whose targets far enough from the source drop's
//      centre take its multipole expansion itself; the direct sums of pairs.cu leave those targets out.
// What it costs: O(L^2) per source and target and O(L^3) per pair of drops instead of the product of
// their node counts. Whole operator applications at 64 drops of degree 16 to 48 (6.6e10 pairs, 95 % of them far), every
// pair directly -> expansions: Laplace double layer FP32 50.4 -> 3.1 ms, stresslet FP32 73.7 -> 9.3 ms, Stokeslet
// double-float 432 -> 27.0 ms; what remains is the direct sums (13.0 ms of the 27.0, 2.2 of the 9.3), the singular
// rows (2.2) and k_far_p2m (4.6, 2.5).
//
// Orders: the truncation error of a pair with source radius a, target radius b and centre distance D is at
// most sum|q| (L+1)^g rho^(L+1) / (D-a-b), rho = max(a/(D-b), b/(D-a)), g the number of derivatives taken; L is
// the smallest order that puts it below 3e-15 (FP64 and double-float sums) or 1e-8 (FP32 sums), one more up to order 24
// in FP64. A pair that would need more than the level's largest order is summed directly.
//
// Errors against sums in 128 bits on the same sources, of a target's sum of magnitudes, expansions and direct sums
// (24 drops of degree 16 to 32, all five kinds, worst of 120 values): FP64 2e-16 and 7e-16, double-float 2.4e-14 and
// 1.4e-12. At the targets where the two differ most, close, elongated and distant drops among them, the expansions'
// error is the smaller one in every kind: FP64 at most 3.8e-16 and 2.2e-15, double-float 6.2e-14 and 1.2e-12.
//
// Arithmetic: native FP64 in FP64 mode, double-float on the FP32 pipe otherwise (a multiply-add costs 12
// FP32 instructions against 64 issue slots), the same code through a template. Harmonics are the real
// orthonormal ones times (r/A)^n with A a power of two above the drop's radius, as
//   kappa_nm Q_nm(2z/A, r^2/A^2) (Re|Im ((x+iy)/A)^m),  Q_n = (2z/A) Q_(n-1) - g_nm (r/A)^2 Q_(n-2), Q_m = 1,
// so that the constants kappa are applied to moments and coefficients and not per node.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <mutex>
#include <vector>

#include "dfloat.cuh"
#include "far.h"
#include "internal.h"

namespace shbim {

namespace {

using dfl::df;

constexpr int kP2mThreads = 256;
constexpr int kP2mTiles = 4;                            // source tiles per CTA
static_assert(kP2mSrc == kP2mThreads * kP2mTiles, "a chunk is a CTA's sources");
constexpr int kL2pWarps = 8;

// ---- arithmetic: double or double-float
__device__ __forceinline__ double t_mul(double a, double b) { return a * b; }
__device__ __forceinline__ df t_mul(df a, df b) { return dfl::mul(a, b); }
__device__ __forceinline__ double t_add(double a, double b) { return a + b; }
__device__ __forceinline__ df t_add(df a, df b) { return dfl::add(a, b); }
__device__ __forceinline__ double t_sub(double a, double b) { return a - b; }
__device__ __forceinline__ df t_sub(df a, df b) { return dfl::sub(a, b); }
__device__ __forceinline__ double t_neg(double a) { return -a; }
__device__ __forceinline__ df t_neg(df a) { return dfl::neg(a); }
__device__ __forceinline__ double t_pow2(double a, float s) { return a * (double)s; }     // s a power of two
__device__ __forceinline__ df t_pow2(df a, float s) { return df{a.hi * s, a.lo * s}; }
__device__ __forceinline__ void t_from(double v, double& o) { o = v; }
__device__ __forceinline__ void t_from(double v, df& o) { o = dfl::from_double(v); }
template <class T>
__device__ __forceinline__ T from_d(double v) {
  T o;
  t_from(v, o);
  return o;
}
__device__ __forceinline__ double t_double(double a) { return a; }
__device__ __forceinline__ double t_double(df a) { return dfl::to_double(a); }

__device__ __forceinline__ float t_float(double a) { return (float)a; }
__device__ __forceinline__ float t_float(df a) { return a.hi; }
// leading FP32 part of an element in memory
__device__ __forceinline__ float f_ld(const double* p, int64_t i) { return (float)p[i]; }
__device__ __forceinline__ float f_ld(const df* p, int64_t i) { return reinterpret_cast<const float*>(p)[2 * i]; }
__device__ __forceinline__ float warp_total_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double t_ld(const double* p, int64_t i) { return p[i]; }
__device__ __forceinline__ df t_ld(const df* p, int64_t i) {
  const float2 v = reinterpret_cast<const float2*>(p)[i];
  return df{v.x, v.y};
}
__device__ __forceinline__ void t_st(double* p, int64_t i, double v) { p[i] = v; }
__device__ __forceinline__ void t_st(df* p, int64_t i, df v) {
  reinterpret_cast<float2*>(p)[i] = make_float2(v.hi, v.lo);
}
// two neighbouring values by one 16-byte load (p + i 16-byte aligned)
__device__ __forceinline__ void t_ld2(const double* p, int64_t i, double& a, double& b) {
  const double2 v = *reinterpret_cast<const double2*>(p + i);
  a = v.x;
  b = v.y;
}
__device__ __forceinline__ void t_ld2(const df* p, int64_t i, df& a, df& b) {
  const float4 v = *reinterpret_cast<const float4*>(p + i);
  a = df{v.x, v.y};
  b = df{v.z, v.w};
}

__device__ __forceinline__ double t_rsqrt(double a) { return rsqrt(a); }
__device__ __forceinline__ df t_rsqrt(df a) { return dfl::rsqrt(a); }

template <class T>
struct Acc;
template <>
struct Acc<double> {
  double v = 0.0;
  __device__ __forceinline__ void add_prod(double a, double b) { v = fma(a, b, v); }
  __device__ __forceinline__ void add(double a) { v += a; }
  __device__ __forceinline__ double value() const { return v; }
};
template <>
struct Acc<df> {
  dfl::acc v;
  __device__ __forceinline__ void add_prod(df a, df b) { v.add_prod(a, b); }
  __device__ __forceinline__ void add(df a) { v.add(a); }
  __device__ __forceinline__ df value() const { return v.value(); }
};

__device__ __forceinline__ double shfl_x(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ df shfl_x(df a, int o) {
  return df{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
template <class T>
__device__ __forceinline__ T warp_total(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = t_add(v, shfl_x(v, o));
  return v;
}

__host__ __device__ __forceinline__ int tri_n(int L) { return (L + 1) * (L + 2) / 2; }
__host__ __device__ __forceinline__ int tri_o(int L, int m) { return m * (L + 1) - m * (m - 1) / 2; }

// (x + i y)^m by binary powers
template <class T>
__device__ void complex_pow(T x, T y, int m, T& c, T& s) {
  T bx = x, by = y;
  bool one = true;
  c = from_d<T>(1.0);
  s = from_d<T>(0.0);
  while (m > 0) {
    if (m & 1) {
      if (one) {
        c = bx;
        s = by;
        one = false;
      } else {
        const T n = t_sub(t_mul(c, bx), t_mul(s, by));
        s = t_add(t_mul(c, by), t_mul(s, bx));
        c = n;
      }
    }
    m >>= 1;
    if (m > 0) {
      const T n = t_sub(t_mul(bx, bx), t_mul(by, by));
      const T p = t_mul(bx, by);
      by = t_add(p, p);
      bx = n;
    }
  }
}

// ---- 1. charges of every source: the strengths themselves (Laplace), f and y.f (single layer), the symmetric
// tensor u_k n_l + n_k u_l and the vector (y.u) n + (y.n) u (double layer)
struct SrcView {
  const double* src;       // FP64 positions, normals
  const float* src32;      // relative to the centres, FP32 and low parts
  const float* src32lo;
  const double* dens;      // FP64 strengths [6][nsource]
  const float* dens32;
  const float* dens32lo;   // null: the FP32 strengths are all there is
  int64_t n;
};

__device__ __forceinline__ void src_get(const SrcView& V, int c, int64_t s, const double* ctr, double& o) {
  o = V.src[c * V.n + s] - (c < 3 ? ctr[c] : 0.0);
}
__device__ __forceinline__ void src_get(const SrcView& V, int c, int64_t s, const double*, df& o) {
  o = df{V.src32[c * V.n + s], V.src32lo[c * V.n + s]};
}
__device__ __forceinline__ void dens_get(const SrcView& V, int c, int64_t s, double& o) { o = V.dens[c * V.n + s]; }
__device__ __forceinline__ void dens_get(const SrcView& V, int c, int64_t s, df& o) {
  o = df{V.dens32[c * V.n + s], V.dens32lo ? V.dens32lo[c * V.n + s] : 0.f};
}
template <class T>
__device__ __forceinline__ T dot3(const T* a, const T* b) {
  return t_add(t_add(t_mul(a[0], b[0]), t_mul(a[1], b[1])), t_mul(a[2], b[2]));
}

template <class T, int MODE>
__global__ void k_far_charges(SrcView V, const DropDev* __restrict__ drops, T* __restrict__ q) {
  const DropDev D = drops[blockIdx.y];
  const double ctr[3] = {D.cx, D.cy, D.cz};
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < D.ns; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = D.src_off + e;
    if (MODE == kFarLap) {
      T v;
      dens_get(V, 0, s, v);
      t_st(q, s, v);
      continue;
    }
    T y[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) src_get(V, c, s, ctr, y[c]);
    int o = 0;
    if (MODE == kFarS || MODE == kFarSD) {
      T f[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dens_get(V, c, s, f[c]);
        t_st(q, (int64_t)c * V.n + s, f[c]);
      }
      t_st(q, 3 * V.n + s, dot3(y, f));
      o = 4;
    }
    if (MODE == kFarD || MODE == kFarSD) {
      T u[3], n[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dens_get(V, 3 + c, s, u[c]);
        src_get(V, 3 + c, s, ctr, n[c]);
      }
      const T yu = dot3(y, u), yn = dot3(y, n);
      const int64_t N = V.n;
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b) {
          const int k = a == 0 ? b : (a == 1 ? 2 + b : 5);
          t_st(q, (o + k) * N + s, t_add(t_mul(u[a], n[b]), t_mul(n[a], u[b])));
        }
#pragma unroll
      for (int c = 0; c < 3; ++c) t_st(q, (o + 6 + c) * N + s, t_add(t_mul(yu, n[c]), t_mul(yn, u[c])));
    }
  }
}

// Moments without their constants: for one chunk of up to 1024 sources of a drop and the orders m = g and
// L - g (together L + 2 columns, so every CTA of a drop has the same work), sums over the chunk of
// q Q_nm (Re|Im (x+iy)^m). Threads first advance the recurrence of their own sources by eight degrees and leave
// Q C and Q S of the tile in shared memory; then warp w sums degree n0 + w over the tile for every charge.
// Degrees above nfull go on in FP32, 16 at a time and two per warp: a far pair's ratio rho is at most 0.608, so
// degree n is rho^n of the result and the FP32 rounding (about n 2^-24, independent from source to source) of
// what nfull leaves out stays below the level's truncation error.
// Bound by instruction issue up to nfull (about 35 + 24 NQ instructions per source and (n, m) in double-float; Stokeslet
// of 24 drops of degree 16 to 32: 2.9 of 4 a cycle, FMA pipe 47 %), above it, where FP32 sums spend most degrees, by the
// latency of the charges' reads at sixteen warps per SM (stresslet: 2.2 a cycle, L1 29 %, 2.3 cycles of waiting for
// memory per issue). Four tiles share one cross-lane reduction.
template <class T, int NQ>
__global__ void __launch_bounds__(kP2mThreads, 2)
k_far_p2m(SrcView V, const DropDev* __restrict__ drops, const FarChunk* __restrict__ chunks, const int* __restrict__ Lsrc,
          int nfull, const float* __restrict__ inv_scale, const T* __restrict__ rec, const T* __restrict__ q,
          T* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char far_smem[];
  T* QC = reinterpret_cast<T*>(far_smem);               // [8][kP2mThreads]
  T* QS = QC + 8 * kP2mThreads;
  float* FC = reinterpret_cast<float*>(far_smem);       // [16][kP2mThreads]
  float* FS = FC + 16 * kP2mThreads;
  const FarChunk ch = chunks[blockIdx.x];
  const int L = Lsrc[ch.drop];
  const int g = blockIdx.y;
  if (2 * g > L) return;                                // uniform over the CTA
  const DropDev D = drops[ch.drop];
  const double ctr[3] = {D.cx, D.cy, D.cz};
  const float inv = inv_scale[ch.drop];
  const int ntri = tri_n(L);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntile = (ch.count + kP2mThreads - 1) / kP2mThreads;
  T* out = part + (int64_t)NQ * 2 * ch.part;
  T z2[kP2mTiles], r2[kP2mTiles], C[kP2mTiles], S[kP2mTiles], q1[kP2mTiles], q2[kP2mTiles];
#pragma unroll
  for (int t = 0; t < kP2mTiles; ++t) {
    const int e = t * kP2mThreads + tid;
    T x = from_d<T>(0.0), y = x, z = x;
    if (e < ch.count) {
      const int64_t s = D.src_off + ch.first + e;
      src_get(V, 0, s, ctr, x);
      src_get(V, 1, s, ctr, y);
      src_get(V, 2, s, ctr, z);
      x = t_pow2(x, inv);
      y = t_pow2(y, inv);
      z = t_pow2(z, inv);
    }
    z2[t] = t_pow2(z, 2.f);
    r2[t] = t_add(t_add(t_mul(x, x), t_mul(y, y)), t_mul(z, z));
  }
  for (int half = 0; half < 2; ++half) {
    const int m = half == 0 ? g : L - g;
    if (half == 1 && m == g) break;
#pragma unroll
    for (int t = 0; t < kP2mTiles; ++t) {
      const int e = t * kP2mThreads + tid;
      C[t] = S[t] = from_d<T>(0.0);
      if (e < ch.count) {
        const int64_t s = D.src_off + ch.first + e;
        T x, y;
        src_get(V, 0, s, ctr, x);
        src_get(V, 1, s, ctr, y);
        complex_pow(t_pow2(x, inv), t_pow2(y, inv), m, C[t], S[t]);
      }
      q1[t] = from_d<T>(1.0);
      q2[t] = from_d<T>(0.0);
    }
    const T* rc = rec + tri_o(kFarLmax, m) - m;
    int n0 = m;
    for (; n0 <= min(L, nfull); n0 += 8) {
      Acc<T> ac[NQ], as[NQ];
      const int nn = min(8, L + 1 - n0);
#pragma unroll
      for (int t = 0; t < kP2mTiles; ++t) {
        if (t >= ntile) break;
        __syncthreads();
        for (int k = 0; k < nn; ++k) {
          const int n = n0 + k;
          if (n > m) {
            // Q_n from Q_(n-1) (q1) and Q_(n-2) (q2)
            T v = t_mul(z2[t], q1[t]);
            if (n > m + 1) v = t_sub(v, t_mul(t_mul(t_ld(rc, n), r2[t]), q2[t]));
            q2[t] = q1[t];
            q1[t] = v;
          }
          t_st(QC, k * kP2mThreads + tid, t_mul(q1[t], C[t]));
          t_st(QS, k * kP2mThreads + tid, t_mul(q1[t], S[t]));
        }
        __syncthreads();
        if (warp < nn) {
          const T* qt = q + D.src_off + ch.first + t * kP2mThreads;
          const int cnt = min(kP2mThreads, ch.count - t * kP2mThreads);
          for (int e = lane; e < cnt; e += 32) {
            const T c = t_ld(QC, warp * kP2mThreads + e), sn = t_ld(QS, warp * kP2mThreads + e);
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
              const T w = t_ld(qt, (int64_t)k * V.n + e);
              ac[k].add_prod(c, w);
              as[k].add_prod(sn, w);
            }
          }
        }
      }
      if (warp < nn) {
        T* o = out + tri_o(L, m) + n0 + warp - m;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
          const T a = warp_total(ac[k].value()), b = warp_total(as[k].value());
          if (lane == 0) {
            t_st(o, (int64_t)(2 * k) * ntri, a);
            t_st(o, (int64_t)(2 * k + 1) * ntri, b);
          }
        }
      }
    }
    if (n0 > L) continue;
    float fz[kP2mTiles], fr[kP2mTiles], fc[kP2mTiles], fs[kP2mTiles], f1[kP2mTiles], f2[kP2mTiles];
#pragma unroll
    for (int t = 0; t < kP2mTiles; ++t) {
      fz[t] = t_float(z2[t]);
      fr[t] = t_float(r2[t]);
      fc[t] = t_float(C[t]);
      fs[t] = t_float(S[t]);
      f1[t] = t_float(q1[t]);
      f2[t] = t_float(q2[t]);
    }
    for (; n0 <= L; n0 += 16) {
      float a0[NQ], a1[NQ], b0[NQ], b1[NQ];
#pragma unroll
      for (int k = 0; k < NQ; ++k) a0[k] = a1[k] = b0[k] = b1[k] = 0.f;
      const int nn = min(16, L + 1 - n0);
#pragma unroll
      for (int t = 0; t < kP2mTiles; ++t) {
        if (t >= ntile) break;
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
          const int n = n0 + k;
          if (n > m && n <= L) {
            float v = fz[t] * f1[t];
            if (n > m + 1) v = fmaf(-f_ld(rc, n) * fr[t], f2[t], v);
            f2[t] = f1[t];
            f1[t] = v;
          }
          FC[k * kP2mThreads + tid] = n <= L ? f1[t] * fc[t] : 0.f;
          FS[k * kP2mThreads + tid] = n <= L ? f1[t] * fs[t] : 0.f;
        }
        __syncthreads();
        if (2 * warp < nn) {
          const T* qt = q + D.src_off + ch.first + t * kP2mThreads;
          const int cnt = min(kP2mThreads, ch.count - t * kP2mThreads);
          const float* c0 = FC + 2 * warp * kP2mThreads;
          const float* s0 = FS + 2 * warp * kP2mThreads;
          for (int e = lane; e < cnt; e += 32) {
            const float x0 = c0[e], x1 = c0[kP2mThreads + e], y0 = s0[e], y1 = s0[kP2mThreads + e];
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
              const float w = f_ld(qt, (int64_t)k * V.n + e);
              a0[k] = fmaf(x0, w, a0[k]);
              a1[k] = fmaf(x1, w, a1[k]);
              b0[k] = fmaf(y0, w, b0[k]);
              b1[k] = fmaf(y1, w, b1[k]);
            }
          }
        }
      }
      if (2 * warp < nn) {
        T* o = out + tri_o(L, m) + n0 + 2 * warp - m;
        const bool two = 2 * warp + 1 < nn;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
          const float c0 = warp_total_f(a0[k]), c1 = warp_total_f(a1[k]);
          const float s0 = warp_total_f(b0[k]), s1 = warp_total_f(b1[k]);
          if (lane == 0) {
            t_st(o, (int64_t)(2 * k) * ntri, from_d<T>((double)c0));
            t_st(o, (int64_t)(2 * k + 1) * ntri, from_d<T>((double)s0));
            if (two) {
              t_st(o, (int64_t)(2 * k) * ntri + 1, from_d<T>((double)c1));
              t_st(o, (int64_t)(2 * k + 1) * ntri + 1, from_d<T>((double)s1));
            }
          }
        }
      }
    }
  }
}

// chunks of a drop added in order, times kappa: coefficient (n, m) of every charge, [drop][charge][(L+1)^2]
template <class T>
__global__ void k_far_vsum(const FarSrcDrop* __restrict__ sd, const int* __restrict__ Lsrc, int nq,
                           const T* __restrict__ kap, const T* __restrict__ part, T* __restrict__ v) {
  const int j = blockIdx.y;
  const int L = Lsrc[j];
  if (L < 0) return;
  const FarSrcDrop d = sd[j];
  const int ntri = tri_n(L), nc = (L + 1) * (L + 1);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nq * nc; e += gridDim.x * blockDim.x) {
    const int k = e / nc, i = e - k * nc;
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    const int mm = i - n * n - n, m = abs(mm);
    const int cs = mm < 0 ? 1 : 0;
    Acc<T> a;
    int64_t o = (int64_t)nq * 2 * d.part + (int64_t)(2 * k + cs) * ntri + tri_o(L, m) + n - m;
    for (int c = 0; c < d.nchunk; ++c, o += (int64_t)nq * 2 * ntri) a.add(t_ld(part, o));
    t_st(v, (int64_t)nq * d.coef + (int64_t)k * nc + i, t_mul(a.value(), t_ld(kap, tri_o(kFarLmax, m) + n - m)));
  }
}

template <class T>
__device__ __forceinline__ T coef_at(const T* __restrict__ c, int n, int m) { return t_ld(c, n * n + n + m); }

// sum_c p_c . grad: moment (n, m) of dipoles from the charge-like moments v_c of their components
template <class T>
__device__ T dipole_moment(const T* __restrict__ vx, const T* __restrict__ vy, const T* __restrict__ vz, int n, int mm,
                           const T* __restrict__ la, const T* __restrict__ lp, const T* __restrict__ lq) {
  Acc<T> a;
  if (n == 0) return a.value();
  const int m = abs(mm), sg = mm < 0 ? -1 : 1, k = n - 1;
  const int t = tri_o(kFarLmax, m) + n - m;
  const T P = t_ld(lp, t), Q = t_ld(lq, t);
  if (m <= k) a.add_prod(t_ld(la, t), coef_at(vz, k, mm));
  if (mm == 0) {
    if (k >= 1) {
      a.add_prod(P, coef_at(vx, k, 1));
      a.add_prod(P, coef_at(vy, k, -1));
    }
    return a.value();
  }
  if (m + 1 <= k) {
    a.add_prod(P, coef_at(vx, k, sg * (m + 1)));
    a.add_prod(sg > 0 ? P : t_neg(P), coef_at(vy, k, -sg * (m + 1)));
  }
  // toward m - 1: the sine of order zero does not exist
  if (sg > 0 || m >= 2) a.add_prod(t_neg(Q), coef_at(vx, k, sg * (m - 1)));
  if (sg < 0)
    a.add_prod(t_neg(Q), coef_at(vy, k, m - 1));
  else if (m >= 2)
    a.add_prod(Q, coef_at(vy, k, -(m - 1)));
  return a.value();
}

// moments of the four potentials of the Stokes kernels with dipoles (modes D and SD)
template <class T, int MODE>
__global__ void k_far_dipoles(const FarSrcDrop* __restrict__ sd, const int* __restrict__ Lsrc,
                              const float* __restrict__ inv_scale, const T* __restrict__ la, const T* __restrict__ lp,
                              const T* __restrict__ lq, const T* __restrict__ v, T* __restrict__ mom) {
  constexpr int NQ = MODE == kFarD ? 9 : 13, O = MODE == kFarD ? 0 : 4;
  const int j = blockIdx.y;
  const int L = Lsrc[j];
  if (L < 0) return;
  const FarSrcDrop d = sd[j];
  const int nc = (L + 1) * (L + 1);
  const T* vj = v + (int64_t)NQ * d.coef;
  T* mj = mom + 4 * d.coef;
  const T w = from_d<T>((double)inv_scale[j] / 6.0);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 4 * nc; e += gridDim.x * blockDim.x) {
    const int k = e / nc, i = e - k * nc;
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    const int mm = i - n * n - n;
    // component c of the moment vector: tensor row k (xx xy xz yy yz zz), or the vector for psi
    const int c0 = k == 3 ? 6 : k, c1 = k == 3 ? 7 : (k == 0 ? 1 : k + 2), c2 = k == 3 ? 8 : (k == 0 ? 2 : k + 3);
    T r = t_mul(w, dipole_moment(vj + (int64_t)(O + c0) * nc, vj + (int64_t)(O + c1) * nc, vj + (int64_t)(O + c2) * nc,
                                 n, mm, la, lp, lq));
    if (MODE == kFarSD) r = t_add(r, t_ld(vj, (int64_t)k * nc + i));
    t_st(mj, (int64_t)k * nc + i, r);
  }
}

// ---- 2. translation of one potential of one far pair
// Dz by -+alpha in place on all degrees of X: (x[m], x[-m]) turned by m alpha
template <class T>
__device__ __forceinline__ void far_dz(T* X, int nc, const T* c, const T* s, bool neg) {
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    const int m = i - n * n - n;
    if (m <= 0) continue;
    const T a = t_ld(X, i), b = t_ld(X, i - 2 * m);
    const T cm = t_ld(c, m);
    T sm = t_ld(s, m);
    if (neg) sm = t_neg(sm);
    t_st(X, i, t_sub(t_mul(cm, a), t_mul(sm, b)));
    t_st(X, i - 2 * m, t_add(t_mul(sm, a), t_mul(cm, b)));
  }
}

// Y = Dq X (or Dq^T X) degree by degree: nonzeros of a row are every second element from start
template <class T>
__device__ __forceinline__ void far_dq(const T* X, T* Y, int nc, const T* __restrict__ val, const int* __restrict__ off,
                                       const int2* __restrict__ pat) {
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    const int w = 2 * n + 1;
    const int2 p = pat[i];                 // start, count
    const T* x = X + n * n + p.x;
    int64_t o = off[n] + (i - n * n);
    Acc<T> a;
    for (int k = 0; k < p.y; ++k, o += w) a.add_prod(t_ld(val, o), t_ld(x, 2 * k));
    t_st(Y, i, a.value());
  }
}

// One CTA per (far pair, potential): all in shared memory; O(2 L^3) multiply-adds. Rotations cost as much as the
// translation (Dq has a quarter of its entries); tables are read from L1 along consecutive rows. Bound by L1 (46 to 52 %)
// and waiting: 1.9 to 2.5 instructions a cycle, barriers between short loops 1.4 to 4.5 cycles per issue, memory 4.
template <class T>
__global__ void __launch_bounds__(256)
k_far_m2l(const FarPair* __restrict__ pairs, int npot, const FarSrcDrop* __restrict__ sd, const int* __restrict__ Lsrc,
          const double* __restrict__ ang, FarTab<T> tab, const T* __restrict__ mom, int64_t out0, T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char far_smem[];
  const FarPair p = pairs[blockIdx.x];
  const int L = p.L, n1 = L + 1, nc = n1 * n1;
  T* X = reinterpret_cast<T*>(far_smem);
  T* Y = X + nc;
  T* a = Y + nc;                            // [6][n1]
  for (int i = threadIdx.x; i < 6 * n1; i += blockDim.x) t_st(a, i, from_d<T>(ang[p.ang + i / n1 * p.na + i % n1]));
  const int Ls = Lsrc[p.j];
  const int64_t ncs = (int64_t)(Ls + 1) * (Ls + 1);
  const T* M = mom + npot * sd[p.j].coef + blockIdx.y * ncs;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) t_st(X, i, t_ld(M, i));
  __syncthreads();
  far_dz(X, nc, a, a + n1, true);
  __syncthreads();
  far_dq(X, Y, nc, tab.dq_r, tab.dq_off, tab.pat_r);
  __syncthreads();
  far_dz(Y, nc, a + 2 * n1, a + 3 * n1, true);
  __syncthreads();
  far_dq(Y, X, nc, tab.dq_c, tab.dq_off, tab.pat_c);
  __syncthreads();
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    t_st(X, i, t_mul(t_ld(X, i), t_ld(a, 4 * n1 + n)));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int l = (int)sqrtf((float)i);
    while (l * l > i) --l;
    while ((l + 1) * (l + 1) <= i) ++l;
    const int mm = i - l * l - l, m = abs(mm);
    int64_t o = tab.tr_off[l] + m;
    Acc<T> s;
    for (int n = m; n <= L; ++n, o += l + 1) s.add_prod(t_ld(tab.tr, o), t_ld(X, n * n + n + mm));
    T v = t_mul(s.value(), t_ld(a, 5 * n1 + l));
    if ((l + m) & 1) v = t_neg(v);
    t_st(Y, i, v);
  }
  __syncthreads();
  far_dq(Y, X, nc, tab.dq_r, tab.dq_off, tab.pat_r);
  __syncthreads();
  far_dz(X, nc, a + 2 * n1, a + 3 * n1, false);
  __syncthreads();
  far_dq(X, Y, nc, tab.dq_c, tab.dq_off, tab.pat_c);
  __syncthreads();
  far_dz(Y, nc, a, a + n1, false);
  __syncthreads();
  T* dst = out + npot * (p.out - out0) + (int64_t)blockIdx.y * nc;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) t_st(dst, i, t_ld(Y, i));
}

// ---- 3. local expansions
// Sum over the far drops of a target drop, in order; psi is moved to the target drop's centre. A CTA lays out 32 pairs at
// a time (their place and shift, whose FP64 differences would otherwise be formed by every thread), and a thread has the
// terms of four of them in flight: one pair after the other, each a chain of three loads, the stresslet of 1024 drops of
// degree 4 took 12.9 ms here (7.9 so, in five parts), of 64 drops of degree 16 0.20 (0.05), in double-float.
constexpr int kLsumThreads = 128;
template <class T>
__global__ void __launch_bounds__(kLsumThreads)
k_far_lsum(const FarTgtDrop* __restrict__ td, const FarPair* __restrict__ pairs, const DropDev* __restrict__ drops, int npot,
           int drop0, int64_t out0, const T* __restrict__ lp, T* __restrict__ loc) {
  constexpr int kTile = 32, kFly = 4;
  __shared__ int s_nc[kTile];
  __shared__ int64_t s_out[kTile];
  __shared__ __align__(8) unsigned char s_shift[3 * kTile * 8];
  T* shift = reinterpret_cast<T*>(s_shift);
  const int i = drop0 + blockIdx.y;
  const FarTgtDrop d = td[i];
  const int nc = (d.L + 1) * (d.L + 1);
  if (d.L < 0 || blockIdx.x * kLsumThreads >= npot * nc) return;    // the whole CTA
  const int e = blockIdx.x * kLsumThreads + threadIdx.x;
  const int k = e / nc, c = e - k * nc;
  const bool mine = e < npot * nc;
  Acc<T> s;
  for (int p0 = d.pair0; p0 < d.pair1; p0 += kTile) {
    const int n = min(kTile, d.pair1 - p0);
    __syncthreads();
    if (threadIdx.x < n) {
      const FarPair q = pairs[p0 + threadIdx.x];
      s_nc[threadIdx.x] = (q.L + 1) * (q.L + 1);
      s_out[threadIdx.x] = npot * (q.out - out0);
      if (npot == 4) {
        const DropDev Di = drops[q.i], Dj = drops[q.j];
        t_st(shift, threadIdx.x, from_d<T>(Dj.cx - Di.cx));
        t_st(shift, kTile + threadIdx.x, from_d<T>(Dj.cy - Di.cy));
        t_st(shift, 2 * kTile + threadIdx.x, from_d<T>(Dj.cz - Di.cz));
      }
    }
    __syncthreads();
    if (!mine) continue;
    for (int u0 = 0; u0 < n; u0 += kFly) {
      T v[kFly], w[kFly][3];
      bool in[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const int ncp = u0 + u < n ? s_nc[u0 + u] : 0;
        in[u] = c < ncp;
        v[u] = w[u][0] = w[u][1] = w[u][2] = from_d<T>(0.0);
        if (!in[u]) continue;
        const T* l = lp + s_out[u0 + u];
        v[u] = t_ld(l, (int64_t)k * ncp + c);
        if (k == 3)
#pragma unroll
          for (int a = 0; a < 3; ++a) w[u][a] = t_ld(l, (int64_t)a * ncp + c);
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        if (!in[u]) continue;
        s.add(v[u]);
        if (k == 3)
#pragma unroll
          for (int a = 0; a < 3; ++a) s.add_prod(t_ld(shift, a * kTile + u0 + u), w[u][a]);
      }
    }
  }
  if (mine) t_st(loc, npot * d.coef + (int64_t)k * nc + c, s.value());
}

// coefficient (n', mu) of the derivative along axis ax of the expansion l of order L (without 1/B)
template <class T>
__device__ T grad_coef(const T* __restrict__ l, int L, int n1, int mu, int ax, const T* __restrict__ la,
                       const T* __restrict__ lp, const T* __restrict__ lq) {
  Acc<T> a;
  const int n = n1 + 1, m = abs(mu);
  if (n > L) return a.value();
  const bool sn = mu < 0;
  if (ax == 2) {
    a.add_prod(t_ld(la, tri_o(kFarLmax, m) + n - m), coef_at(l, n, mu));
    return a.value();
  }
  // from order m - 1 (factor lp) and from order m + 1 (factor lq) of degree n
  const T Q = t_ld(lq, tri_o(kFarLmax, m + 1) + n - m - 1);
  if (ax == 0) {
    if (m >= 1 && (!sn || m >= 2)) a.add_prod(t_ld(lp, tri_o(kFarLmax, m - 1) + n - m + 1), coef_at(l, n, sn ? -(m - 1) : m - 1));
    a.add_prod(t_neg(Q), coef_at(l, n, sn ? -(m + 1) : m + 1));
  } else if (!sn) {
    a.add_prod(t_neg(Q), coef_at(l, n, -(m + 1)));
    if (m >= 2) a.add_prod(t_neg(t_ld(lp, tri_o(kFarLmax, m - 1) + n - m + 1)), coef_at(l, n, -(m - 1)));
  } else {
    a.add_prod(t_ld(lp, tri_o(kFarLmax, m - 1) + n - m + 1), coef_at(l, n, m - 1));
    a.add_prod(Q, coef_at(l, n, m + 1));
  }
  return a.value();
}

// expansions the targets evaluate, times kappa, interleaved: [(m, n)][set][cos, sin]
// sets: SL value; DL gradient; Stokes phi_i + d_i psi (3), d_i phi_k (9, k major)
template <class T, int NS>
__global__ void k_far_lset(const FarTgtDrop* __restrict__ td, const float* __restrict__ inv_scale, FarTab<T> tab,
                           int npot, const T* __restrict__ loc, T* __restrict__ set) {
  const int i = blockIdx.y;
  const FarTgtDrop d = td[i];
  if (d.L < 0) return;
  const int L = d.L, nc = (L + 1) * (L + 1), ntri = tri_n(L);
  const T* l = loc + npot * d.coef;
  const T inv = from_d<T>((double)inv_scale[i]);
  T* out = set + (int64_t)2 * NS * d.tri;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ntri * 2 * NS; e += gridDim.x * blockDim.x) {
    const int o = e / (2 * NS), r = e - o * 2 * NS;
    const int st = r >> 1, cs = r & 1;
    int m = 0;
    while (m < L && tri_o(L, m + 1) <= o) ++m;
    const int n = m + (o - tri_o(L, m));
    T v = from_d<T>(0.0);
    if (!(cs == 1 && m == 0)) {
      const int mu = cs ? -m : m;
      if (NS == 1) {
        v = coef_at(l, n, mu);
      } else if (NS == 3) {
        v = t_mul(inv, grad_coef(l, L, n, mu, st, tab.la, tab.lp, tab.lq));
      } else if (st < 3) {
        v = t_add(coef_at(l + (int64_t)st * nc, n, mu),
                  t_mul(inv, grad_coef(l + (int64_t)3 * nc, L, n, mu, st, tab.la, tab.lp, tab.lq)));
      } else {
        const int k = (st - 3) / 3, ax = (st - 3) - 3 * k;
        v = t_mul(inv, grad_coef(l + (int64_t)k * nc, L, n, mu, ax, tab.la, tab.lp, tab.lq));
      }
      v = t_mul(v, t_ld(tab.kap, tri_o(kFarLmax, m) + n - m));
    }
    t_st(out, e, v);
  }
}

// ---- 4. values at the targets: a CTA takes 32 targets of one drop (one per lane), its eight warps the orders
// m = w, w + 8, ... The coefficients of the next degrees are read by the lanes side by side while the present ones
// are used from a slot of shared memory, as broadcasts (read where they are used, they cost two L2 latencies per
// degree: 4.7 ms instead of 1.0 for the Stokes sets at 1.4e5 targets). Degrees above nfull in FP32, as for the
// moments. Bound by issue and the latency of the recurrence's chain (35 + 24 NS instructions per target and (n, m) in
// double-float; 2.6 of 4 a cycle, FMA pipe 50 %, for FP32 sums 1.9 and 33 %); splitting the orders keeps every SM busy
// from a few thousand targets on.
template <class T, int NS>
__device__ __forceinline__ void eval_sets(T x, T y, T z, int L, int Ls, int nfull, const T* __restrict__ rec,
                                          const T* __restrict__ set, T* __restrict__ red, unsigned char* slot_raw) {
  constexpr int VB = 2 * NS;               // coefficients of one (n, m)
  constexpr int NB = 32 / VB;              // degrees per slot
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T z2 = t_pow2(z, 2.f);
  const T r2 = t_add(t_add(t_mul(x, x), t_mul(y, y)), t_mul(z, z));
  T* slot = reinterpret_cast<T*>(slot_raw) + warp * 64;
  float* fslot = reinterpret_cast<float*>(slot);
  T* tot = red + (warp * NS) * 32 + lane;               // [NS] with stride 32: this thread's own totals
#pragma unroll
  for (int k = 0; k < NS; ++k) t_st(tot, k * 32, from_d<T>(0.0));
  T C, S, C8, S8;
  complex_pow(x, y, warp, C, S);
  complex_pow(x, y, kL2pWarps, C8, S8);
  int buf = 0;
  for (int m = warp; m <= L; m += kL2pWarps) {
    T q1 = from_d<T>(1.0), q2 = from_d<T>(0.0);
    const T* c = set + (int64_t)VB * tri_o(Ls, m);
    const T* rc = rec + tri_o(kFarLmax, m) - m;
    const int left = (L - m + 1) * VB;
    int o = 0, n = m;
    T nx = (lane < NB * VB && lane < left) ? t_ld(c, lane) : from_d<T>(0.0);
    if (m <= nfull) {
      Acc<T> ac[NS], as[NS];
      for (; n <= min(L, nfull); n += NB) {
        const T* sl = slot + buf * 32;
        t_st(slot + buf * 32, lane, nx);
        __syncwarp();
        buf ^= 1;
        o += NB * VB;
        nx = (lane < NB * VB && o + lane < left) ? t_ld(c, o + lane) : from_d<T>(0.0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
          if (n + i > L) break;
          if (n + i > m) {
            T v = t_mul(z2, q1);
            if (n + i > m + 1) v = t_sub(v, t_mul(t_mul(t_ld(rc, n + i), r2), q2));
            q2 = q1;
            q1 = v;
          }
#pragma unroll
          for (int k = 0; k < NS; ++k) {
            T a, bb;
            t_ld2(sl, i * VB + 2 * k, a, bb);
            ac[k].add_prod(a, q1);
            as[k].add_prod(bb, q1);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        Acc<T> s;
        s.add(t_ld(tot, k * 32));
        s.add_prod(C, ac[k].value());
        s.add_prod(S, as[k].value());
        t_st(tot, k * 32, s.value());
      }
    }
    if (n <= L) {
      float f1 = t_float(q1), f2 = t_float(q2);
      const float fz = t_float(z2), fr = t_float(r2);
      float fa[NS], fb[NS];
#pragma unroll
      for (int k = 0; k < NS; ++k) fa[k] = fb[k] = 0.f;
      for (; n <= L; n += NB) {
        const float* sl = fslot + buf * 64;
        fslot[buf * 64 + lane] = t_float(nx);
        __syncwarp();
        buf ^= 1;
        o += NB * VB;
        nx = (lane < NB * VB && o + lane < left) ? t_ld(c, o + lane) : from_d<T>(0.0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
          if (n + i > L) break;
          if (n + i > m) {
            float v = fz * f1;
            if (n + i > m + 1) v = fmaf(-f_ld(rc, n + i) * fr, f2, v);
            f2 = f1;
            f1 = v;
          }
#pragma unroll
          for (int k = 0; k < NS; ++k) {
            fa[k] = fmaf(sl[i * VB + 2 * k], f1, fa[k]);
            fb[k] = fmaf(sl[i * VB + 2 * k + 1], f1, fb[k]);
          }
        }
      }
      const float fC = t_float(C), fS = t_float(S);
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        Acc<T> s;
        s.add(t_ld(tot, k * 32));
        s.add(from_d<T>((double)fmaf(fC, fa[k], fS * fb[k])));
        t_st(tot, k * 32, s.value());
      }
    }
    const T nC = t_sub(t_mul(C, C8), t_mul(S, S8));
    S = t_add(t_mul(C, S8), t_mul(S, C8));
    C = nC;
  }
  __syncthreads();
  for (int k = warp; k < NS; k += kL2pWarps) {
    Acc<T> s;
#pragma unroll
    for (int w = 0; w < kL2pWarps; ++w) s.add(t_ld(red, (w * NS + k) * 32 + lane));
    t_st(red, k * 32 + lane, s.value());    // slot (0, k) is read by this thread only
  }
  __syncthreads();
}

template <class T, int NS>
__global__ void __launch_bounds__(32 * kL2pWarps, 2)
k_far_l2p(const FarTgtDrop* __restrict__ td, const int2* __restrict__ blocks, const DropDev* __restrict__ drops,
          const float* __restrict__ inv_scale, int nfull, const T* __restrict__ rec, const T* __restrict__ set,
          const double* __restrict__ tgt, int64_t ntarget, double* __restrict__ out) {
  __shared__ __align__(16) unsigned char red_raw[kL2pWarps * NS * 32 * 8];
  __shared__ __align__(16) unsigned char slot_raw[kL2pWarps * 2 * 32 * 8];
  T* red = reinterpret_cast<T*>(red_raw);
  const int2 b = blocks[blockIdx.x];                    // drop, first target within the drop
  const FarTgtDrop d = td[b.x];
  const DropDev D = drops[b.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool ok = b.y + lane < D.nt;
  const int64_t t = D.tgt_off + (ok ? b.y + lane : 0);
  const float inv = inv_scale[b.x];
  const T x = t_pow2(from_d<T>(tgt[t] - D.cx), inv), y = t_pow2(from_d<T>(tgt[ntarget + t] - D.cy), inv),
          z = t_pow2(from_d<T>(tgt[2 * ntarget + t] - D.cz), inv);
  eval_sets<T, NS>(x, y, z, d.L, d.L, nfull, rec, set + (int64_t)2 * NS * d.tri, red, slot_raw);
  if (!ok) return;
  const double w4 = 0.07957747154594766788;
  if (NS == 1) {
    if (warp == 0) out[t] += w4 * t_double(t_ld(red, lane));
  } else if (NS == 3) {
    if (warp == 0) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(tgt[(3 + k) * ntarget + t], t_double(t_ld(red, k * 32 + lane)), v);
      out[t] -= w4 * v;
    }
  } else if (warp < 3) {
    const int c = warp;
    const double B = 1.0 / (double)inv;     // a power of two
    const T xs[3] = {x, y, z};
    Acc<T> g;
#pragma unroll
    for (int k = 0; k < 3; ++k) g.add_prod(xs[k], t_ld(red, (3 + 3 * k + c) * 32 + lane));
    const double v = t_double(t_ld(red, c * 32 + lane)) - B * t_double(g.value());
    out[3 * D.tgt_off + (int64_t)c * D.nt + (t - D.tgt_off)] += w4 * v;
  }
}


// ---- 5. close pairs: targets far enough from the source drop's centre take its multipole expansion itself,
// Phi = 1/r sum_nm c_nm R_nm(x A / r^2), the regular harmonics at the inverted point, so the sets and the
// evaluation are those of the local expansions. A drop's neighbours at gaps of 0.2 to 1 have half to two thirds of
// their targets beyond 1.7 to 2 radii, and a value of order 45 costs a seventh to a thirtieth of a sum over the
// 5e3 to 2e4 sources of a drop of degree 24 to 48.

// coefficient (n, mm) of the derivative along axis ax of the multipole expansion v, times -A (a dipole along ax)
template <class T>
__device__ T multi_grad(const T* __restrict__ v, int n, int mm, int ax, const T* __restrict__ la,
                        const T* __restrict__ lp, const T* __restrict__ lq) {
  Acc<T> a;
  if (n == 0) return a.value();
  const int m = abs(mm), sg = mm < 0 ? -1 : 1, k = n - 1;
  const int t = tri_o(kFarLmax, m) + n - m;
  if (ax == 2) {
    if (m <= k) a.add_prod(t_ld(la, t), coef_at(v, k, mm));
    return a.value();
  }
  const T Pv = t_ld(lp, t), Q = t_ld(lq, t);
  if (mm == 0) {
    if (k >= 1) a.add_prod(Pv, coef_at(v, k, ax == 0 ? 1 : -1));
    return a.value();
  }
  if (ax == 0) {
    if (m + 1 <= k) a.add_prod(Pv, coef_at(v, k, sg * (m + 1)));
    if (sg > 0 || m >= 2) a.add_prod(t_neg(Q), coef_at(v, k, sg * (m - 1)));
  } else {
    if (m + 1 <= k) a.add_prod(sg > 0 ? Pv : t_neg(Pv), coef_at(v, k, -sg * (m + 1)));
    if (sg < 0)
      a.add_prod(t_neg(Q), coef_at(v, k, m - 1));
    else if (m >= 2)
      a.add_prod(Q, coef_at(v, k, -(m - 1)));
  }
  return a.value();
}

// the sets of k_far_lset of a source drop's multipole expansion
template <class T, int NS>
__global__ void k_far_mset(const FarSrcDrop* __restrict__ sd, const int* __restrict__ Lsrc,
                           const float* __restrict__ inv_scale, FarTab<T> tab, int npot, const T* __restrict__ mom,
                           T* __restrict__ set) {
  const int j = blockIdx.y;
  const int L = Lsrc[j];
  if (L < 0) return;
  const FarSrcDrop d = sd[j];
  const int nc = (L + 1) * (L + 1), ntri = tri_n(L);
  const T* l = mom + npot * d.coef;
  const T inv = from_d<T>(-(double)inv_scale[j]);
  T* out = set + (int64_t)2 * NS * d.tri;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ntri * 2 * NS; e += gridDim.x * blockDim.x) {
    const int o = e / (2 * NS), r = e - o * 2 * NS;
    const int st = r >> 1, cs = r & 1;
    int m = 0;
    while (m < L && tri_o(L, m + 1) <= o) ++m;
    const int n = m + (o - tri_o(L, m));
    T v = from_d<T>(0.0);
    if (!(cs == 1 && m == 0)) {
      const int mu = cs ? -m : m;
      if (NS == 1) {
        v = coef_at(l, n, mu);
      } else if (NS == 3) {
        v = t_mul(inv, multi_grad(l, n, mu, st, tab.la, tab.lp, tab.lq));
      } else if (st < 3) {
        v = t_add(coef_at(l + (int64_t)st * nc, n, mu),
                  t_mul(inv, multi_grad(l + (int64_t)3 * nc, n, mu, st, tab.la, tab.lp, tab.lq)));
      } else {
        const int k = (st - 3) / 3, ax = (st - 3) - 3 * k;
        v = t_mul(inv, multi_grad(l + (int64_t)k * nc, n, mu, ax, tab.la, tab.lp, tab.lq));
      }
      v = t_mul(v, t_mul(t_ld(tab.kap, tri_o(kFarLmax, m) + n - m), from_d<T>(12.566370614359172954 / (2 * n + 1))));
    }
    t_st(out, e, v);
  }
}

// values of one entry's expansion at one group of targets, [group][component][32]; bound as k_far_l2p
template <class T, int NS>
__global__ void __launch_bounds__(32 * kL2pWarps, 2)
k_far_m2p(int nent, const int* __restrict__ ent_tgt, NearList nl, const FarSrcDrop* __restrict__ sd,
          const int* __restrict__ Lsrc, const DropDev* __restrict__ drops, const float* __restrict__ inv_scale, int nfull,
          const T* __restrict__ rec, const T* __restrict__ set, const double* __restrict__ tgt, int64_t ntarget,
          double* __restrict__ part) {
  constexpr int NC = NS == 12 ? 3 : 1;
  __shared__ __align__(16) unsigned char red_raw[kL2pWarps * NS * 32 * 8];
  __shared__ __align__(16) unsigned char slot_raw[kL2pWarps * 2 * 32 * 8];
  T* red = reinterpret_cast<T*>(red_raw);
  const int64_t f = blockIdx.x;
  const int en = entry_of(nl.goff, nent, f);
  const int j = nl.drop[en];
  const DropDev Dj = drops[j];
  const int g = (int)(f - nl.goff[en]);
  if (nl.direct(en, g, Dj.ns)) return;                  // uniform over the CTA
  const DropDev Di = drops[ent_tgt[en]];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sl = g * kFarGroup + lane;
  const int64_t t = nl.tgt[Di.tgt_off + min(sl, Di.nt - 1)];
  const float inv = inv_scale[j];
  const T x = t_pow2(from_d<T>(tgt[t] - Dj.cx), inv), y = t_pow2(from_d<T>(tgt[ntarget + t] - Dj.cy), inv),
          z = t_pow2(from_d<T>(tgt[2 * ntarget + t] - Dj.cz), inv);
  const T ri = t_rsqrt(t_add(t_add(t_mul(x, x), t_mul(y, y)), t_mul(z, z)));
  const T ri2 = t_mul(ri, ri);
  eval_sets<T, NS>(t_mul(x, ri2), t_mul(y, ri2), t_mul(z, ri2), nl.order[f], Lsrc[j], nfull, rec,
                   set + (int64_t)2 * NS * sd[j].tri, red, slot_raw);
  const double w = 0.07957747154594766788 * (double)inv * t_double(ri);
  double* o = part + f * NC * 32 + lane;
  if (NS == 1) {
    if (warp == 0) o[0] = w * t_double(t_ld(red, lane));
  } else if (NS == 3) {
    if (warp == 0) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(tgt[(3 + k) * ntarget + t], t_double(t_ld(red, k * 32 + lane)), v);
      o[0] = -w * v;
    }
  } else if (warp < 3) {
    const int c = warp;
    const T xs[3] = {x, y, z};
    Acc<T> a;
#pragma unroll
    for (int k = 0; k < 3; ++k) a.add_prod(xs[k], t_ld(red, (3 + 3 * k + c) * 32 + lane));
    o[32 * c] = w * (t_double(t_ld(red, c * 32 + lane)) - t_double(a.value()) / (double)inv);
  }
}

// a drop's targets: the entries' values in order
template <int NC>
__global__ void k_far_msum(NearList nl, const DropDev* __restrict__ drops, const double* __restrict__ part,
                           double* __restrict__ out) {
  const int i = blockIdx.y;
  const DropDev D = drops[i];
  const int sl = blockIdx.x * blockDim.x + threadIdx.x;
  if (sl >= D.nt) return;
  const int g = sl / kFarGroup;
  double s[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) s[c] = 0.0;
  for (unsigned en = nl.off[i]; en < nl.off[i + 1] - 1; ++en) {
    if (nl.direct(en, g, drops[nl.drop[en]].ns)) continue;
    const double* p = part + (nl.goff[en] + g) * NC * 32 + (sl & 31);
#pragma unroll
    for (int c = 0; c < NC; ++c) s[c] += p[32 * c];
  }
  const int64_t t = nl.tgt[D.tgt_off + sl] - D.tgt_off;
#pragma unroll
  for (int c = 0; c < NC; ++c) out[(int64_t)NC * D.tgt_off + (int64_t)c * D.nt + t] += s[c];
}

// ---- constants (host, once per process; copied to each context's device memory)
struct FarHost {
  std::vector<double> dq_r, dq_c, tr, kap, rec, la, lp, lq;
  std::vector<int> dq_off, tr_off;
  std::vector<int2> pat_r, pat_c;
};

const FarHost& far_host() {
  static FarHost H;
  static std::once_flag once;
  std::call_once(once, [] {
    const int L = kFarLmax;
    const int nt = tri_n(L);
    // Dq_n: real-basis matrix of Rx(pi/2) from d^n(pi/2) (recursion of Trapani and Navaza, 2006) with the phases
    // of the z-rotations by +-pi/2
    std::vector<double> prev(1, 1.0);
    H.dq_off.assign(L + 2, 0);
    for (int n = 0; n <= L; ++n) H.dq_off[n + 1] = H.dq_off[n] + (n / 2 + 1) * (2 * n + 1);
    H.dq_r.assign(H.dq_off[L + 1], 0.0);
    H.dq_c.assign(H.dq_off[L + 1], 0.0);
    H.pat_r.resize((size_t)(L + 1) * (L + 1));
    H.pat_c.resize((size_t)(L + 1) * (L + 1));
    for (int l = 0; l <= L; ++l) {
      const int w = 2 * l + 1;
      std::vector<double> d((size_t)w * w, 0.0);
      auto at = [&](int a, int b) -> double& { return d[(size_t)(a + l) * w + b + l]; };
      if (l == 0) {
        d[0] = 1.0;
      } else {
        const int pw = 2 * l - 1;
        auto pr = [&](int a, int b) { return prev[(size_t)(a + l - 1) * pw + b + l - 1]; };
        at(0, l) = -std::sqrt((2.0 * l - 1.0) / (2.0 * l)) * pr(0, l - 1);
        for (int a = 1; a <= l; ++a)
          at(a, l) = std::sqrt(0.5 * l * (2.0 * l - 1.0) / ((double)(l + a) * (l + a - 1))) * pr(a - 1, l - 1);
        for (int a = 0; a <= l; ++a)
          for (int m = l - 1; m >= 0; --m) {
            double v = 2.0 * a / std::sqrt((double)(l - m) * (l + m + 1)) * at(a, m + 1);
            if (m + 2 <= l)
              v -= std::sqrt((double)(l - m - 1) * (l + m + 2) / ((double)(l - m) * (l + m + 1))) * at(a, m + 2);
            at(a, m) = v;
          }
        for (int a = 0; a <= l; ++a)
          for (int m = 0; m <= l; ++m) {
            const double v = at(a, m);
            at(a, -m) = ((l + a) & 1) ? -v : v;
            at(-a, m) = ((l + m) & 1) ? -v : v;
            at(-a, -m) = ((a + m) & 1) ? -v : v;
          }
      }
      prev = d;
      // real basis: S = T Y with S_m = (Y_m + (-1)^m Y_-m)/sqrt2, S_-m = (Y_m - (-1)^m Y_-m)/(i sqrt2)
      using cd = std::complex<double>;
      auto row = [&](int a, int idx[2], cd c[2]) {   // nonzeros of row a of T
        const int m = std::abs(a);
        const double r = std::sqrt(0.5), sg = (m & 1) ? -1.0 : 1.0;
        if (a == 0) {
          idx[0] = 0;
          c[0] = 1.0;
          return 1;
        }
        idx[0] = m;
        idx[1] = -m;
        if (a > 0) {
          c[0] = r;
          c[1] = sg * r;
        } else {
          c[0] = cd(0.0, -r);
          c[1] = cd(0.0, sg * r);
        }
        return 2;
      };
      auto ipow = [](int m) {
        static const cd t[4] = {cd(1, 0), cd(0, 1), cd(-1, 0), cd(0, -1)};
        return t[((m % 4) + 4) % 4];
      };
      std::vector<double> A((size_t)w * w);
      for (int a = -l; a <= l; ++a)
        for (int b = -l; b <= l; ++b) {
          int ia[2], ib[2];
          cd ca[2], cb[2];
          const int na = row(a, ia, ca), nb = row(b, ib, cb);
          cd s = 0.0;
          for (int x = 0; x < na; ++x)
            for (int y = 0; y < nb; ++y) s += ca[x] * ipow(ia[x]) * at(ia[x], ib[y]) * ipow(-ib[y]) * std::conj(cb[y]);
          A[(size_t)(a + l) * w + b + l] = s.real();
        }
      for (int tr = 0; tr < 2; ++tr)
        for (int a = 0; a < w; ++a) {
          auto el = [&](int b) { return tr ? A[(size_t)b * w + a] : A[(size_t)a * w + b]; };
          // the nonzeros of a row are the orders of one sign and one parity
          int big = 0;
          for (int b = 1; b < w; ++b)
            if (std::fabs(el(b)) > std::fabs(el(big))) big = b;
          const int par = std::abs(big - l) & 1;
          int start, count;
          if (big >= l) {
            start = l + par;
            count = (l - par) / 2 + 1;
          } else {
            const int hi = ((l & 1) == par) ? l : l - 1, lo = par ? 1 : 2;   // |m| from lo to hi
            start = l - hi;
            count = (hi - lo) / 2 + 1;
          }
          (tr ? H.pat_c : H.pat_r)[(size_t)l * l + a] = make_int2(start, count);
          for (int k = 0; k < count; ++k) (tr ? H.dq_c : H.dq_r)[H.dq_off[l] + (size_t)k * w + a] = el(start + 2 * k);
        }
    }
    // translation factors (n+l)! / sqrt((n-m)!(n+m)!(l-m)!(l+m)!) 2^-(n+l), laid out [l][n - m][m]
    std::vector<double> lf(2 * L + 2, 0.0);
    for (int k = 2; k <= 2 * L + 1; ++k) lf[k] = lf[k - 1] + std::log((double)k);
    H.tr_off.assign(L + 2, 0);
    for (int l = 0; l <= L; ++l) H.tr_off[l + 1] = H.tr_off[l] + (L + 1) * (l + 1);
    H.tr.assign(H.tr_off[L + 1], 0.0);
    for (int l = 0; l <= L; ++l)
      for (int m = 0; m <= l; ++m) {
        // by ratios from n = m: exact to rounding, where exponentials of logarithms lose digits
        double v = 1.0;   // (m+l)! / sqrt(0! (2m)! (l-m)! (l+m)!) 2^-(m+l) = sqrt(prod (l+m)!/((2m)!(l-m)!)) 2^-(m+l)
        {
          // binomial(l+m, 2m) times 4^-(l+m), factor by factor
          double b = 1.0;
          for (int k = 1; k <= l - m; ++k) b *= (double)(2 * m + k) / k;
          v = std::sqrt(b) * std::ldexp(1.0, -(m + l));
        }
        for (int n = m; n <= L; ++n) {
          if (n > m) v *= 0.5 * (n + l) / std::sqrt((double)(n - m) * (n + m));
          H.tr[H.tr_off[l] + (size_t)(n - m) * (l + 1) + m] = v;
        }
      }
    H.kap.assign(nt, 0.0);
    H.rec.assign(nt, 0.0);
    H.la.assign(nt, 0.0);
    H.lp.assign(nt, 0.0);
    H.lq.assign(nt, 0.0);
    double cm = 1.0 / std::sqrt(4.0 * kPi);
    for (int m = 0; m <= L; ++m) {
      if (m > 0) cm *= -std::sqrt((2.0 * m + 1.0) / (2.0 * m));
      double k = cm * (m > 0 ? kSqrt2 : 1.0);
      for (int n = m; n <= L; ++n) {
        const int o = tri_o(L, m) + n - m;
        const double n2 = (double)n * n, m2 = (double)m * m;
        if (n > m) k *= 0.5 * std::sqrt((4.0 * n2 - 1.0) / (n2 - m2));
        H.kap[o] = k;
        if (n > m + 1) H.rec[o] = 4.0 * ((n - 1.0) * (n - 1.0) - m2) / (4.0 * (n - 1.0) * (n - 1.0) - 1.0);
        if (n > 0) {
          const double f = (2.0 * n + 1.0) / (2.0 * n - 1.0);
          H.la[o] = std::sqrt(f * (n - m) * (n + m));
          H.lp[o] = std::sqrt(f * (n - m) * (n - m - 1.0)) * (m == 0 ? std::sqrt(0.5) : 0.5);
          if (n - m - 1 < 0) H.lp[o] = 0.0;
          H.lq[o] = m == 0 ? 0.0 : std::sqrt(f * (n + m) * (n + m - 1.0)) * (m == 1 ? std::sqrt(0.5) : 0.5);
        }
      }
    }
  });
  return H;
}

}  // namespace

int far_grow(shbim_ctx* ctx, void** p, size_t* cap, size_t bytes, const char* what) {
  if (bytes <= *cap) return SHBIM_OK;
  cudaFree(*p);
  *p = nullptr;
  *cap = 0;
  if (cudaMalloc(p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return fail(ctx, SHBIM_ERR_NOMEM, std::string("cudaMalloc ") + what);
  }
  *cap = bytes;
  return SHBIM_OK;
}

int far_tables(shbim_ctx* ctx) {
  FarState& F = *ctx->far;
  if (F.tables) return SHBIM_OK;
  const FarHost& H = far_host();
  const std::vector<const std::vector<double>*> v{&H.dq_r, &H.dq_c, &H.tr, &H.kap, &H.rec, &H.la, &H.lp, &H.lq};
  size_t n = 0;
  for (auto* a : v) n += a->size();
  const size_t ni = H.dq_off.size() + H.tr_off.size() + 2 * (H.pat_r.size() + H.pat_c.size());
  const size_t bytes = 2 * n * sizeof(double) + (ni + 8) * sizeof(int);
  std::vector<unsigned char> blob(bytes, 0);
  double* hd = reinterpret_cast<double*>(blob.data());
  float2* hf = reinterpret_cast<float2*>(hd + n);
  int* hi = reinterpret_cast<int*>(hf + n);
  unsigned char* dev = nullptr;
  if (cudaMalloc(&dev, bytes) != cudaSuccess) return fail(ctx, SHBIM_ERR_NOMEM, "cudaMalloc expansion tables");
  double* dd = reinterpret_cast<double*>(dev);
  df* ddf = reinterpret_cast<df*>(dd + n);
  int* di = reinterpret_cast<int*>(ddf + n);
  const double** pd[8] = {&F.td.dq_r, &F.td.dq_c, &F.td.tr, &F.td.kap, &F.td.rec, &F.td.la, &F.td.lp, &F.td.lq};
  const df** pf[8] = {&F.tf.dq_r, &F.tf.dq_c, &F.tf.tr, &F.tf.kap, &F.tf.rec, &F.tf.la, &F.tf.lp, &F.tf.lq};
  size_t o = 0;
  for (int k = 0; k < 8; ++k) {
    for (size_t e = 0; e < v[k]->size(); ++e) {
      const double x = (*v[k])[e];
      hd[o + e] = x;
      const float h = (float)x;
      hf[o + e] = make_float2(h, (float)(x - (double)h));
    }
    *pd[k] = dd + o;
    *pf[k] = ddf + o;
    o += v[k]->size();
  }
  size_t q = 0;
  // the int2 patterns first (8-byte aligned)
  std::memcpy(hi + q, H.pat_r.data(), H.pat_r.size() * sizeof(int2));
  F.td.pat_r = F.tf.pat_r = reinterpret_cast<const int2*>(di + q);
  q += 2 * H.pat_r.size();
  std::memcpy(hi + q, H.pat_c.data(), H.pat_c.size() * sizeof(int2));
  F.td.pat_c = F.tf.pat_c = reinterpret_cast<const int2*>(di + q);
  q += 2 * H.pat_c.size();
  std::memcpy(hi + q, H.dq_off.data(), H.dq_off.size() * sizeof(int));
  F.td.dq_off = F.tf.dq_off = di + q;
  q += H.dq_off.size();
  std::memcpy(hi + q, H.tr_off.data(), H.tr_off.size() * sizeof(int));
  F.td.tr_off = F.tf.tr_off = di + q;
  if (cudaMemcpy(dev, blob.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(dev);
    return cuda_fail(ctx, cudaGetLastError(), "copy expansion tables");
  }
  F.tables = dev;
  return SHBIM_OK;
}

namespace {

// degrees carried in full precision: above it rho^n has taken the term below what FP32 loses, whose rounding (about
// n 2^-24, independent from source to source) leaves at the largest ratios of a level 0.608^13 13 2^-24 = 1.2e-9 above
// degree 12 of FP32 sums and 0.578^37 37 2^-24 = 3.4e-15 above degree 36 of double-float ones; FP64 carries all
int far_full(const shbim_ctx* ctx) {
  return ctx->opts.precision == SHBIM_PREC_FP32_COMP ? 12 : (ctx->opts.precision == SHBIM_PREC_DF64 ? 36 : kFarLmax);
}

template <class T>
FarTab<T>& tab_of(FarState& F);
template <>
FarTab<double>& tab_of<double>(FarState& F) { return F.td; }
template <>
FarTab<df>& tab_of<df>(FarState& F) { return F.tf; }

template <class T, int MODE, int NQ>
int expand(shbim_ctx* ctx, const FarPlan& P, int kind, cudaStream_t s) {
  FarState& F = *ctx->far;
  const FarTab<T>& tab = tab_of<T>(F);
  constexpr int npot = MODE == kFarLap ? 1 : 4;
  const bool lo = ctx->opts.precision == SHBIM_PREC_DF64;
  const SrcView V{ctx->geo.src, ctx->geo.src32, ctx->geo.src32lo, ctx->dens_up, ctx->dens_up32, lo ? ctx->dens_up32lo : nullptr,
                  ctx->nsource};
  T* q = static_cast<T*>(F.q);
  T* part = static_cast<T*>(F.part);
  T* v = static_cast<T*>(F.v);
  T* lp = static_cast<T*>(F.lpair);
  T* loc = static_cast<T*>(F.loc);
  T* set = static_cast<T*>(F.set);
  int maxns = 0;
  for (const auto& d : ctx->drops) maxns = std::max(maxns, d.ns);
  const unsigned nd = (unsigned)ctx->n_drops;
  k_far_charges<T, MODE><<<dim3((unsigned)std::min(64, (maxns + 255) / 256), nd), 256, 0, s>>>(V, ctx->drops_dev, q);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_charges");
  const int smem = 2 * 8 * kP2mThreads * 8;
  k_far_p2m<T, NQ><<<dim3((unsigned)P.nchunks, (unsigned)(P.lmax / 2 + 1)), kP2mThreads, smem, s>>>(
      V, ctx->drops_dev, P.chunks, P.Lsrc, far_full(ctx), F.inv_src, tab.rec, q, part);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_p2m");
  const int ncm = (P.lmax + 1) * (P.lmax + 1);
  k_far_vsum<T><<<dim3((unsigned)((NQ * ncm + 255) / 256), nd), 256, 0, s>>>(P.sd, P.Lsrc, NQ, tab.kap, part, v);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_vsum");
  const T* mom = v;
  if constexpr (MODE == kFarD || MODE == kFarSD) {
    k_far_dipoles<T, MODE><<<dim3((unsigned)((4 * ncm + 255) / 256), nd), 256, 0, s>>>(
        P.sd, P.Lsrc, F.inv_src, tab.la, tab.lp, tab.lq, v, static_cast<T*>(F.mom));
    SHBIM_CHECK_LAUNCH(ctx, "k_far_dipoles");
    mom = static_cast<T*>(F.mom);
  }
  const int sm = (2 * ncm + 6 * (P.lmax + 1)) * 8;
  constexpr int sm_max = (2 * (kFarCapMax + 1) * (kFarCapMax + 1) + 6 * (kFarCapMax + 1)) * 8;
  SHBIM_CUDA(ctx, cudaFuncSetAttribute(k_far_m2l<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_max));
  for (const FarBatch& b : P.batches) {
    if (b.pair1 > b.pair0) {
      k_far_m2l<T><<<dim3((unsigned)(b.pair1 - b.pair0), npot), 256, sm, s>>>(P.pairs + b.pair0, npot, P.sd, P.Lsrc,
                                                                            F.ang, tab, mom, b.out0, lp);
      SHBIM_CHECK_LAUNCH(ctx, "k_far_m2l");
    }
    k_far_lsum<T><<<dim3((unsigned)((npot * ncm + kLsumThreads - 1) / kLsumThreads), (unsigned)(b.drop1 - b.drop0)), kLsumThreads,
                    0, s>>>(
        P.td, P.pairs, ctx->drops_dev, npot, b.drop0, b.out0, lp, loc);
    SHBIM_CHECK_LAUNCH(ctx, "k_far_lsum");
  }
  const unsigned lb = (unsigned)((tri_n(P.lmax) * 2 * kSets[kind] + 127) / 128);
  if (kind == 1)
    k_far_lset<T, 1><<<dim3(lb, nd), 128, 0, s>>>(P.td, F.inv_tgt, tab, npot, loc, set);
  else if (kind == 0)
    k_far_lset<T, 3><<<dim3(lb, nd), 128, 0, s>>>(P.td, F.inv_tgt, tab, npot, loc, set);
  else
    k_far_lset<T, 12><<<dim3(lb, nd), 128, 0, s>>>(P.td, F.inv_tgt, tab, npot, loc, set);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_lset");
  if (far_near(ctx, P, kind).order) {
    T* ms = static_cast<T*>(F.mset);
    if (kind == 1)
      k_far_mset<T, 1><<<dim3(lb, nd), 128, 0, s>>>(P.sd, P.Lsrc, F.inv_src, tab, npot, mom, ms);
    else if (kind == 0)
      k_far_mset<T, 3><<<dim3(lb, nd), 128, 0, s>>>(P.sd, P.Lsrc, F.inv_src, tab, npot, mom, ms);
    else
      k_far_mset<T, 12><<<dim3(lb, nd), 128, 0, s>>>(P.sd, P.Lsrc, F.inv_src, tab, npot, mom, ms);
    SHBIM_CHECK_LAUNCH(ctx, "k_far_mset");
  }
  return SHBIM_OK;
}

template <class T, int NS>
int evaluate_multi(shbim_ctx* ctx, const FarPlan& P, int kind, double* out, cudaStream_t s) {
  constexpr int NC = NS == 12 ? 3 : 1;
  FarState& F = *ctx->far;
  const NearList nl = far_near(ctx, P, kind);
  if (!nl.order) return SHBIM_OK;
  double* part = static_cast<double*>(F.mpart);
  k_far_m2p<T, NS><<<(unsigned)P.ngroup, 32 * kL2pWarps, 0, s>>>(P.nent, P.ent_tgt, nl, P.sd, P.Lsrc, ctx->drops_dev, F.inv_src,
                                                               far_full(ctx), tab_of<T>(F).rec, static_cast<const T*>(F.mset),
                                                               ctx->geo.tgt, ctx->ntarget, part);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_m2p");
  int maxnt = 0;
  for (const auto& d : ctx->drops) maxnt = std::max(maxnt, d.nt);
  k_far_msum<NC><<<dim3((unsigned)((maxnt + 127) / 128), (unsigned)ctx->n_drops), 128, 0, s>>>(nl, ctx->drops_dev, part, out);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_msum");
  return SHBIM_OK;
}

template <class T>
int expand_kind(shbim_ctx* ctx, const FarPlan& P, int kind, cudaStream_t s) {
  if (kind < 2) return expand<T, kFarLap, 1>(ctx, P, kind, s);
  if (kind == 3) return expand<T, kFarS, 4>(ctx, P, kind, s);
  if (kind == 4) return expand<T, kFarD, 9>(ctx, P, kind, s);
  return expand<T, kFarSD, 13>(ctx, P, kind, s);
}

template <class T>
int evaluate_kind(shbim_ctx* ctx, const FarPlan& P, int kind, double* out, cudaStream_t s) {
  FarState& F = *ctx->far;
  const FarTab<T>& tab = tab_of<T>(F);
  const T* set = static_cast<const T*>(F.set);
  const unsigned g = (unsigned)P.nblocks, b = 32 * kL2pWarps;
  if (kind == 1)
    k_far_l2p<T, 1><<<g, b, 0, s>>>(P.td, P.blocks, ctx->drops_dev, F.inv_tgt, far_full(ctx), tab.rec, set, ctx->geo.tgt, ctx->ntarget, out);
  else if (kind == 0)
    k_far_l2p<T, 3><<<g, b, 0, s>>>(P.td, P.blocks, ctx->drops_dev, F.inv_tgt, far_full(ctx), tab.rec, set, ctx->geo.tgt, ctx->ntarget, out);
  else
    k_far_l2p<T, 12><<<g, b, 0, s>>>(P.td, P.blocks, ctx->drops_dev, F.inv_tgt, far_full(ctx), tab.rec, set, ctx->geo.tgt, ctx->ntarget, out);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_l2p");
  return kind == 1   ? evaluate_multi<T, 1>(ctx, P, kind, out, s)
         : kind == 0 ? evaluate_multi<T, 3>(ctx, P, kind, out, s)
                     : evaluate_multi<T, 12>(ctx, P, kind, out, s);
}

}  // namespace

int far_expand(shbim_ctx* ctx, const FarPlan& P, int kind, cudaStream_t s) {
  return ctx->opts.precision == SHBIM_PREC_FP64 ? expand_kind<double>(ctx, P, kind, s) : expand_kind<df>(ctx, P, kind, s);
}

int far_evaluate(shbim_ctx* ctx, const FarPlan& P, int kind, double* out, cudaStream_t s) {
  return ctx->opts.precision == SHBIM_PREC_FP64 ? evaluate_kind<double>(ctx, P, kind, out, s)
                                                : evaluate_kind<df>(ctx, P, kind, out, s);
}

}  // namespace shbim
