// Legendre stage of the analysis of the singular-row weights (Section 2.1) on the fifth-generation
// tensor cores, with FP64-class accuracy:
//   v[item][n^2 + n +- m] = s_m sum_j F[(cs, m)][item][j] Pbar_n^m(t_j),   s_0 = 1, s_m = sqrt(2),
// the cosine part (cs = 0) giving order +m and the sine part (cs = 1) order -m. For one (cs, m) it
// is a GEMM of the items' latitude rows (the Fourier stage's output, order-major) by the fixed
// table Pbar_n^m(t_j), n = m .. p; both are split into six bfloat16 digits (tc.cuh) for drops up to degree 39 and
// seven above (whose other stages are double-float, 2^-44), the table per row n after its own power-of-two scale.
//
// Work decomposition: persistent CTAs (one per SM, sixteen producer warps and one MMA warp) take contiguous ranges
// of work items (cs, m, tile of 64 degrees, 128 items) ordered by m, so the table of one m (up to 130 KB) is
// loaded once per CTA and order. The 128 rows of an item are contiguous in memory: eight lanes read a row's 128 bytes
// per K step side by side and hold the whole row in registers, find its scale by shuffles and write the digit
// planes of one K step of 16 latitudes after the other into one of two stages; the next item's rows are requested
// before the products of this one are waited for. The MMA warp issues a row digit against up to
// four table digits at once. The epilogue combines the accumulators and scatters the outputs into the coefficient rows.
// Bound by latency and the digit arithmetic. Reading the rows by thread (one row per thread) took 24 us per item at
// degree 32, most of it in uncoalesced reads. Drops of degree 48 and 64 (3.1e9 row values): 151 ms on the FP32 pipe, each
// item rereading the whole table from L2; 29 ms here. Every wait is bounded; a timeout sets the error flag and the
// CTA stops.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"
#include "tc.cuh"

namespace shbim {

namespace {

using dfl::df;
using namespace tc;

constexpr int kProducers = 512;
constexpr int kThreads = kProducers + 32;
constexpr int kNtile = 64;                     // degrees per tile (7 x 64 tensor-memory columns)
constexpr int kKmax = 144;                     // latitudes q + 1 = 2p + 2 <= 130, padded
static_assert(diag_sums_exact(kKmax) && diag_sums_exact7(kKmax), "Legendre stage: digit sums must stay exact in FP32");
constexpr int kPlaneA = kMT * kKS;
constexpr uint32_t kTmemCols = 512;

__host__ __device__ inline int padded16(int w) { return w <= 16 ? 16 : (w + 15) / 16 * 16; }
__host__ __device__ inline int leg_digits_of(int p) { return p <= 39 ? kDig : kDig7; }
inline int leg_ksteps(int p) { return (2 * p + 2 + kKS - 1) / kKS; }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// units (m, degree tile, cs) in the order of m, tile, cs; the sine part of m = 0 does not exist. Work item it -> unit
// it / tiles, item tile it % tiles. Orders with more than 64 degrees (m = 0 of p = 64) have two degree tiles.
struct LegItems {
  int p, tiles, over;            // over: orders with two degree tiles (p + 1 - m > 64)
  int64_t total;
  __host__ __device__ LegItems(int p_, int64_t nitems) : p(p_) {
    tiles = (int)((nitems + kMT - 1) / kMT);
    over = p + 1 > kNtile ? p + 1 - kNtile : 0;
    total = (int64_t)(2 * (p + 1) - 1 + (over > 0 ? 2 * over - 1 : 0)) * tiles;
  }
  __host__ __device__ void decode(int64_t it, int& m, int& nt, int& cs, int& tile) const {
    int u = (int)(it / tiles);
    tile = (int)(it - (int64_t)u * tiles);
    m = nt = cs = 0;
    const int first = over > 0 ? 2 : 1;        // units of m = 0
    if (u < first) {
      nt = u;
      return;
    }
    u -= first;
    const int heavy = over > 1 ? 4 * (over - 1) : 0;   // m = 1 .. over - 1: two degree tiles, cos and sin
    if (u < heavy) {
      m = 1 + (u >> 2);
      nt = (u >> 1) & 1;
      cs = u & 1;
      return;
    }
    u -= heavy;
    m = (over > 1 ? over : 1) + (u >> 1);
    cs = u & 1;
  }
};

// the table of (m, nt) is index m for the first degree tile, p + 1 + m for the second
__host__ __device__ inline int leg_slot(int p, int m, int nt) { return nt * (p + 1) + m; }

template <int KS, int ND>
__global__ void __launch_bounds__(kThreads, 1)
k_leg_tc(const float2* __restrict__ FT, int64_t nitems, int p, const uint4* __restrict__ tdig,
         const int* __restrict__ toff, const signed char* __restrict__ texp, float2* __restrict__ coef,
         int64_t coef_stride, int table_bytes, int* __restrict__ err, uint64_t wlim) {
  // dynamic shared memory: [the current order's table planes][two stages of row digit planes]
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[2];
  __shared__ __align__(8) uint64_t empty[2];
  __shared__ __align__(8) uint64_t tbar;
  __shared__ uint32_t tmem_base;
  __shared__ int rowexp[kMT];
  __shared__ int colexp[kNtile];
  const int K = 2 * p + 2;                       // latitudes of the degree 2p + 1 grid
  const int P1 = p + 1;
  uint8_t* sB = smem;
  uint8_t* sA = smem + table_bytes;
  const int tid = threadIdx.x, warp = tid >> 5;
  const bool producer = tid < kProducers;
  const LegItems I(p, nitems);
  const int64_t per = (I.total + gridDim.x - 1) / gridDim.x;
  const int64_t it0 = (int64_t)blockIdx.x * per, it1 = min(I.total, it0 + per);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    mbar_init(&full[0], kProducers / 32);
    mbar_init(&full[1], kProducers / 32);
    mbar_init(&empty[0], 1);
    mbar_init(&empty[1], 1);
    mbar_init(&tbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = tmem_base;
  uint32_t uses[2] = {0u, 0u};
  uint32_t tphase = 0u;
  bool tpend = false;        // a table copy issued and not yet waited for (MMA thread)
  int cur = -1;
  bool abort_all = false;
  const int r_loc = (tid >> 3) & 63, piece = tid & 7;   // row within a half tile, 16-byte piece of a K step
  const int64_t nrowsF = nitems * K;             // values of one (cs, m) slice of F
  // rows r_loc and 64 + r_loc of a work item, every K step: two latitudes per 16-byte load (K is even, so a pair lies
  // wholly inside or wholly past the row)
  float4 v[2][KS];
  auto load_item = [&](int64_t it) {
    int m, nt, cs, tile;
    I.decode(it, m, nt, cs, tile);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t item = (int64_t)tile * kMT + 64 * h + r_loc;
      const bool ok = item < nitems;
      const float2* row = FT + (int64_t)(cs * P1 + m) * nrowsF + (ok ? item : 0) * K;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int k = ks * kKS + 2 * piece;
        v[h][ks] = ok && k < K ? *reinterpret_cast<const float4*>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  if (producer && it0 < it1) load_item(it0);
  for (int64_t it = it0; it < it1 && !abort_all; ++it) {
    int m, nt, cs, tile;
    I.decode(it, m, nt, cs, tile);
    const int Nm = min(kNtile, P1 - m - nt * kNtile), Np = padded16(Nm);
    // a new table (after every product of the previous one has completed, which the previous item's epilogue
    // waited for) and its row exponents
    const int slot = leg_slot(p, m, nt);
    if (slot != cur) {
      if (tid == kProducers) {
        bulk_load(sB, tdig + toff[slot], (uint32_t)(KS * ND * Np * kKS * 2), &tbar);
        tpend = true;
      }
      if (tid < Nm) colexp[tid] = texp[slot * kNtile + tid];
      cur = slot;
    }
    bool bad = false;
    if (producer) {
      // power-of-two scale of a row, max |hi| < 2^e, over its eight lanes
      float sc[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float mx = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) mx = fmaxf(mx, fmaxf(fabsf(v[h][ks].x), fabsf(v[h][ks].z)));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        int e = 0;
        frexpf(mx, &e);
        e = max(e, -120);
        sc[h] = __int_as_float((127 + 7 - e) << 23);
        if (piece == 0) rowexp[64 * h + r_loc] = e;
      }
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int st = ks & 1;
        if (!bad && uses[st] > 0 && !mbar_wait(&empty[st], (uses[st] - 1) & 1, wlim)) bad = true;
        bad = __any_sync(0xffffffffu, bad);      // a warp goes on or stops together
        if (bad) continue;
        uint8_t* base = sA + st * (ND * kPlaneA * 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float d0[ND], d1[ND];
          digits_n<ND>(v[h][ks].x * sc[h], v[h][ks].y * sc[h], d0);
          digits_n<ND>(v[h][ks].z * sc[h], v[h][ks].w * sc[h], d1);
          const int off = canon16(64 * h + r_loc, 2 * piece) * 2;
#pragma unroll
          for (int j = 0; j < ND; ++j)
            *reinterpret_cast<uint32_t*>(base + j * kPlaneA * 2 + off) = pack_bf16f(d0[j], d1[j]);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(&full[st]);
        ++uses[st];
      }
      if (!bad && it + 1 < it1) load_item(it + 1);
    } else if (tid == kProducers) {
      if (tpend) {
        if (!mbar_wait(&tbar, tphase, wlim)) bad = true;
        tphase ^= 1u;
        tpend = false;
      }
      const int gmax = 256 / Np;
      for (int ks = 0; ks < KS && !bad; ++ks) {
        const int st = ks & 1;
        if (!mbar_wait(&full[st], uses[st] & 1, wlim)) {
          bad = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const uint32_t a0 = smem_u32(sA + st * (ND * kPlaneA * 2)), b0 = smem_u32(sB + (size_t)ks * ND * Np * kKS * 2);
        // row digit j_a against up to gmax consecutive table digits (their planes lie one after the other like the rows
        // of one operand, their products go to consecutive accumulators); the products of the top row digit come first
        // and, in the first K step, overwrite all ND accumulators
        for (int ja = ND - 1; ja >= 0; --ja)
          for (int jb = ND - 1 - ja; jb < ND;) {
            const int g = min(gmax, ND - jb);
            const uint32_t acc = (ks > 0 || ja != ND - 1) ? 1u : 0u;
            mma_bf16(tmem + (uint32_t)((ja + jb - (ND - 1)) * Np), desc_k16(a0 + ja * kPlaneA * 2),
                     desc_k16(b0 + jb * Np * kKS * 2), idesc_bf16(Np * g), acc);
            jb += g;
          }
        mma_commit(&empty[st]);
        ++uses[st];
      }
    } else {
      for (int ks = 0; ks < KS; ++ks) ++uses[ks & 1];
    }
    if (__syncthreads_or(bad)) {
      abort_all = true;
      break;
    }
    {
      const int st = (KS - 1) & 1;
      if (__syncthreads_or(!mbar_wait(&empty[st], (uses[st] - 1) & 1, wlim))) {
        abort_all = true;
        break;
      }
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    // epilogue: warp w (< 16) reads lanes 32 (w % 4) .. +31; column blocks of 4 split among w, w + 4, w + 8, w + 12
    if (producer) {
      const int lq = warp & 3, wq = warp >> 2;
      const int rl = 32 * lq + (tid & 31);
      const int64_t ie = (int64_t)tile * kMT + rl;
      const int ee = rowexp[rl];
      const df s2 = m == 0 ? df{1.f, 0.f} : df{1.41421353816986084f, 2.4203234971764687e-08f};   // sqrt 2
      float2* crow = coef + (ie < nitems ? ie : 0) * coef_stride;
      for (int cb = wq; cb < Np / 4; cb += 4) {
        uint32_t a[ND][4];
#pragma unroll
        for (int dg = 0; dg < ND; ++dg)
          tmem_ld4(tmem + ((uint32_t)(32 * lq) << 16) + (uint32_t)(dg * Np + cb * 4), a[dg]);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n");
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int nn = cb * 4 + j;
          if (ie < nitems && nn < Nm) {
            float s[ND];
#pragma unroll
            for (int dg = 0; dg < ND; ++dg) s[dg] = __uint_as_float(a[dg][j]);
            const float2 r = scale2(combine_n<ND>(s), ee + colexp[nn] - 14);
            const df o = dfl::mul(df{r.x, r.y}, s2);
            const int n = m + nt * kNtile + nn;
            crow[n * n + n + (cs ? -m : m)] = make_float2(o.hi, o.lo);
          }
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
  }
  if (abort_all) {
    for (int st = 0; st < 2; ++st)
      if (uses[st] > 0) mbar_wait(&empty[st], (uses[st] - 1) & 1, kDrainNs);
    if (tid == 0) atomicExch(err, 1);
  }
  if (tpend && tid == kProducers) mbar_wait(&tbar, tphase, kDrainNs);
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols));
}

int leg_table_bytes(int p) {
  return leg_ksteps(p) * leg_digits_of(p) * padded16(std::min(p + 1, kNtile)) * kKS * 2;
}

int leg_tc_smem(int p) { return leg_table_bytes(p) + 2 * leg_digits_of(p) * kPlaneA * 2; }

template <int KS, int ND>
int launch(shbim_ctx* ctx, const DegreeTables& T, const float2* FT, int64_t nitems, float2* coef, int64_t coef_stride,
           cudaStream_t s) {
  const int smem = leg_tc_smem(T.p);
  SHBIM_CUDA(ctx, cudaFuncSetAttribute(k_leg_tc<KS, ND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       leg_tc_smem(std::min(64, KS * kKS / 2 - 1))));
  int dev = 0, nsm = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const LegItems I(T.p, nitems);
  const unsigned grid = (unsigned)std::min<int64_t>(I.total, nsm);
  k_leg_tc<KS, ND><<<grid, kThreads, smem, s>>>(FT, nitems, T.p, reinterpret_cast<const uint4*>(T.leg_digits),
                                                T.leg_toff, T.leg_exp, coef, coef_stride, leg_table_bytes(T.p),
                                                ctx->tc_err, ctx->wait_ns);
  SHBIM_CHECK_LAUNCH(ctx, "k_leg_tc");
  return SHBIM_OK;
}

}  // namespace

bool leg_tc_fits(int p) { return 2 * p + 2 <= kKmax && leg_tc_smem(p) + 4096 <= 227 * 1024; }

// Digit planes of Pbar_n^m(t_j) (degree 2p+1 grid latitudes j, n = m .. p) per order m and tile of 64 degrees:
// [K step][digit][Np x 16, K-major canonical], row n split after its own scale 2^-e.
int leg_tc_digits(shbim_ctx* ctx, int p, const std::vector<double>& alf0, DegreeTables& T) {
  if (!leg_tc_fits(p)) return SHBIM_OK;
  const int P1 = p + 1, K = 2 * p + 2, ksteps = leg_ksteps(p), nd = leg_digits_of(p);
  const int nt = P1 * (p + 2) / 2;
  std::vector<int> off(2 * P1, 0);
  size_t total = 0;
  auto width = [&](int slot) { return std::min(kNtile, P1 - slot % P1 - slot / P1 * kNtile); };
  for (int slot = 0; slot < 2 * P1; ++slot) {
    off[slot] = (int)(total / 8);
    if (width(slot) > 0) total += (size_t)ksteps * nd * padded16(width(slot)) * kKS;
  }
  std::vector<uint16_t> h(total, 0);
  std::vector<signed char> ex((size_t)2 * P1 * kNtile, 0);
  for (int slot = 0; slot < 2 * P1; ++slot) {
    const int m = slot % P1, n0 = slot / P1 * kNtile, Nm = width(slot), Np = padded16(std::max(Nm, 1));
    if (Nm <= 0) continue;
    const int tro = m * (p + 1) - m * (m - 1) / 2 + n0;
    std::vector<int> em(Np, 0);
    for (int nn = 0; nn < Nm; ++nn) {
      double mx = 0.0;
      for (int j = 0; j < K; ++j) mx = std::max(mx, std::fabs(alf0[(size_t)j * nt + tro + nn]));
      int e = 0;
      std::frexp(mx, &e);
      em[nn] = std::max(e, -60);
      ex[(size_t)slot * kNtile + nn] = (signed char)em[nn];
    }
    uint16_t* dst = h.data() + (size_t)off[slot] * 8;
    for (int ks = 0; ks < ksteps; ++ks)
      for (int nn = 0; nn < Np; ++nn)
        for (int kk = 0; kk < kKS; ++kk) {
          const int j = ks * kKS + kk;
          const double v = (nn < Nm && j < K) ? alf0[(size_t)j * nt + tro + nn] : 0.0;
          int dg[kDig7];
          digits_host_n(v, em[nn], nd, dg);
          for (int jd = 0; jd < nd; ++jd) dst[((size_t)ks * nd + jd) * Np * kKS + canon16(nn, kk)] = bf16_int(dg[jd]);
        }
  }
  if (cudaMalloc(&T.leg_digits, h.size() * sizeof(uint16_t)) != cudaSuccess ||
      cudaMalloc(&T.leg_toff, off.size() * sizeof(int)) != cudaSuccess || cudaMalloc(&T.leg_exp, ex.size()) != cudaSuccess)
    return fail(ctx, SHBIM_ERR_NOMEM, "cudaMalloc Legendre digit table");
  if (cudaMemcpy(T.leg_digits, h.data(), h.size() * sizeof(uint16_t), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(T.leg_toff, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(T.leg_exp, ex.data(), ex.size(), cudaMemcpyHostToDevice) != cudaSuccess)
    return fail(ctx, SHBIM_ERR_CUDA, "cudaMemcpy Legendre digit table");
  return SHBIM_OK;
}

int analysis_legendre_tc(shbim_ctx* ctx, const DegreeTables& T, const float2* FT, int64_t nitems, float2* coef,
                         int64_t coef_stride, cudaStream_t s) {
  if (nitems <= 0) return SHBIM_OK;
  if (!T.leg_digits) return fail(ctx, SHBIM_ERR_ARG, "Legendre digit table missing");
  if (!ctx->tc_err) {
    if (cudaMalloc(&ctx->tc_err, sizeof(int)) != cudaSuccess)
      return fail(ctx, SHBIM_ERR_NOMEM, "cudaMalloc tensor-core error flag");
    SHBIM_CUDA(ctx, cudaMemsetAsync(ctx->tc_err, 0, sizeof(int), s));
  }
  const bool seven = leg_digits_of(T.p) == kDig7;
  switch (leg_ksteps(T.p)) {
    case 1: return launch<1, kDig>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 2: return launch<2, kDig>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 3: return launch<3, kDig>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 4: return launch<4, kDig>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 5: return launch<5, kDig>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 6: return launch<6, kDig7>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 7: return launch<7, kDig7>(ctx, T, FT, nitems, coef, coef_stride, s);
    case 8: return launch<8, kDig7>(ctx, T, FT, nitems, coef, coef_stride, s);
    default: break;
  }
  return seven ? launch<9, kDig7>(ctx, T, FT, nitems, coef, coef_stride, s)
               : fail(ctx, SHBIM_ERR_ARG, "degree too large for the tensor-core Legendre stage");
}

}  // namespace shbim
