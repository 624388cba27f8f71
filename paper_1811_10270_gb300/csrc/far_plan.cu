// Plans of the expansions between well-separated drops (far.cu): which pairs of drops are far and at what order, which
// kinds of sums the expansions pay for, and the lists the kernels work through.
//
// The pairs of drops are classified on the GPU, a warp per target drop: k_far_count sums up what every plan would come
// to, per drop, and k_far_fill writes the lists of the plans in use. The host sees O(drops) numbers only. One after
// the other on the host, with lists for all plans copied to the device, set_drops took 1.8 s for 2048 drops of degree 4
// (0.42 without expansions in the library), 0.37 so; 64 drops 5.9 and 5.1 ms. The list of every other drop, for the sums
// without expansions, belongs to the layout; implied in the pair sums instead of read, it made the FP32 double layer
// 2 to 6 % slower.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "far.h"
#include "internal.h"

namespace shbim {

namespace {

// largest ratio rho that order L serves, per plan; the reach of close pairs takes the FP32 number below it
struct RhoTab {
  double r[kFarPlans][kFarCapMax + 1];
};
struct RhoReach {
  float r[kFarCapMax + 1];
};

__host__ __device__ constexpr int plan_cap(int pl) { return far_cap(pl / 3); }

const RhoTab& rho_tab() {
  static const RhoTab T = [] {
    RhoTab t{};
    for (int pl = 0; pl < kFarPlans; ++pl)
      for (int L = 0; L <= plan_cap(pl); ++L)
        t.r[pl][L] = std::pow(kFarEps[pl / 3] / std::pow(L + 1.0, pl % 3), 1.0 / (L + 1));
    for (int pl = 0; pl < 3; ++pl)             // FP64
      for (int L = kFarTight; L > 0; --L) t.r[pl][L] = t.r[pl][L - 1];
    return t;
  }();
  return T;
}

// rho of a pair of drops, sources of j and targets of i; infinite where their spheres overlap
__device__ __forceinline__ double far_ratio(const double* __restrict__ centres, const unsigned* __restrict__ ext, int nd, int i,
                                            int j) {
  double d2 = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double c = centres[3 * i + k] - centres[3 * j + k];
    d2 = fma(c, c, d2);
  }
  const double D = sqrt(d2), a = (double)__uint_as_float(ext[j]), b = (double)__uint_as_float(ext[nd + i]);
  if (!(D > a + b)) return INFINITY;
  return fmax(a / (D - b), b / (D - a));
}

// smallest order that serves rho under plan pl, at least 2; -1: none
__device__ __forceinline__ int far_order(const RhoTab& T, int pl, double rho) {
  const int cap = plan_cap(pl);
  if (!(rho <= T.r[pl][cap])) return -1;
  int a = 0, b = cap;
  while (a < b) {
    const int c = (a + b) >> 1;
    if (T.r[pl][c] < rho)
      a = c + 1;
    else
      b = c;
  }
  return max(a, 2);
}

// largest order that any plan gives the pair
__device__ __forceinline__ int far_order_any(const RhoTab& T, double rho) {
  int L = -1;
#pragma unroll
  for (int pl = 0; pl < kFarPlans; ++pl) L = max(L, far_order(T, pl, rho));
  return L;
}

template <class V>
__device__ __forceinline__ V warp_add(V v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// a warp per target drop: its row under every plan, and the largest orders of the source drops
__global__ void k_far_count(const __grid_constant__ RhoTab T, const double* __restrict__ centres,
                            const unsigned* __restrict__ ext, const DropDev* __restrict__ drops, int nd,
                            FarRow* __restrict__ rows, int* __restrict__ lsrc) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= nd) return;
  int far[kFarPlans], lmax[kFarPlans], ang = 0, pairs = 0;
  int64_t out[kFarPlans], src[kFarPlans];
  double cubes[kFarPlans];
#pragma unroll
  for (int pl = 0; pl < kFarPlans; ++pl) {
    far[pl] = 0;
    lmax[pl] = -1;
    out[pl] = src[pl] = 0;
    cubes[pl] = 0.0;
  }
  for (int j = lane; j < nd; j += 32) {
    if (j == i) continue;
    const double rho = far_ratio(centres, ext, nd, i, j);
    const int ns = drops[j].ns;
    int top = -1;
#pragma unroll
    for (int pl = 0; pl < kFarPlans; ++pl) {
      const int L = far_order(T, pl, rho);
      if (L < 0) continue;
      top = max(top, L);
      far[pl]++;
      lmax[pl] = max(lmax[pl], L);
      out[pl] += (L + 1) * (L + 1);
      src[pl] += ns;
      cubes[pl] += 2.0 * L * L * L;
      if (lsrc[pl * nd + j] < L) atomicMax(lsrc + pl * nd + j, L);
    }
    pairs += top >= 0;
    ang += 6 * (top + 1);
  }
  const int64_t nt = drops[i].nt;
#pragma unroll
  for (int pl = 0; pl < kFarPlans; ++pl) {
    FarRow r;
    r.far = warp_add(far[pl]);
    r.ang = 0;
    r.out = warp_add(out[pl]);
    r.pairs = nt * warp_add(src[pl]);
    r.cubes = warp_add(cubes[pl]);
    r.lmax = lmax[pl];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r.lmax = max(r.lmax, __shfl_xor_sync(0xffffffffu, r.lmax, o));
    r.pad = 0;
    if (lane == 0) rows[(int64_t)pl * nd + i] = r;
  }
  FarRow r{};
  r.far = warp_add(pairs);
  r.ang = warp_add(ang);
  if (lane == 0) rows[(int64_t)kFarPlans * nd + i] = r;
}

// lists of a plan; pl kFarPlans: every pair that is far under some plan, with the order its angles need
struct FillPlan {
  int pl;
  const FarTgtDrop* td;
  const unsigned* off;
  FarPair* pairs;
  int *drop, *ent_tgt;
  int64_t *pre, *goff;
};
struct FillPlans {
  FillPlan p[kFarRows];
};

__device__ __forceinline__ int scan_before(int v, int lane) {
  int s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += t;
  }
  return s - v;
}

// the same warp writes its drop's far pairs and its list of the others, in the order of the drops
__global__ void k_far_fill(const __grid_constant__ RhoTab T, const __grid_constant__ FillPlans plans,
                           const double* __restrict__ centres, const unsigned* __restrict__ ext,
                           const DropDev* __restrict__ drops, int nd) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= nd) return;
  const FillPlan& P = plans.p[blockIdx.y];
  const FarTgtDrop d = P.td[i];
  const int groups = (drops[i].nt + kFarGroup - 1) / kFarGroup;
  const unsigned below = (1u << lane) - 1u;
  int64_t pair = d.pair0, out = d.out, ang = d.ang, goff = d.group, pre = 0;
  unsigned entry = P.drop ? P.off[i] : 0;
  for (int j0 = 0; j0 < nd; j0 += 32) {
    const int j = j0 + lane;
    const bool other = j < nd && j != i;
    const double rho = other ? far_ratio(centres, ext, nd, i, j) : INFINITY;
    const int top = far_order_any(T, rho), L = P.pl < kFarPlans ? far_order(T, P.pl, rho) : top;
    const bool far = L >= 0, near = other && !far;
    const unsigned fm = __ballot_sync(0xffffffffu, far), nm = __ballot_sync(0xffffffffu, near);
    const int o = far ? (L + 1) * (L + 1) : 0, g = 6 * (top + 1), ns = near ? drops[j].ns : 0;
    const int ob = scan_before(o, lane), gb = scan_before(g, lane), nb = scan_before(ns, lane);
    if (far) P.pairs[pair + __popc(fm & below)] = FarPair{i, j, L, top + 1, out + ob, ang + gb};
    if (near && P.drop) {
      const int k = __popc(nm & below);
      P.drop[entry + k] = j;
      P.ent_tgt[entry + k] = i;
      P.pre[entry + k] = pre + nb;
      P.goff[entry + k] = goff + (int64_t)k * groups;
    }
    pair += __popc(fm);
    out += __shfl_sync(0xffffffffu, ob + o, 31);
    ang += __shfl_sync(0xffffffffu, gb + g, 31);
    pre += __shfl_sync(0xffffffffu, nb + ns, 31);
    entry += __popc(nm);
    goff += (int64_t)__popc(nm) * groups;
  }
  if (lane || !P.drop) return;
  P.drop[entry] = P.ent_tgt[entry] = -1;      // end of the list, with the total
  P.pre[entry] = pre;
  P.goff[entry] = goff;
  if (i == nd - 1) P.goff[entry + 1] = goff;
}

// 1 / sqrt(2 m + 1)
struct AngTab {
  double r[kFarCapMax + 1];
};

// cos / sin of m phi and m theta, and the powers (2A/D)^n, (2B/D)^l, of every far pair (once per geometry). A thread per
// pair and one product per value: FP64 instructions bound it: sine, cosine and power of every value apart, 100 to
// 200 of them each, took 160 ms for 1024 drops of degree 4 and six plans, the products 4.9 (the plans share them now). The
// rounding of m factors is that of an angle m phi.
__global__ void k_far_angles(const FarPair* __restrict__ pairs, int npairs, const DropDev* __restrict__ drops,
                             const float* __restrict__ inv_src, const float* __restrict__ inv_tgt,
                             const __grid_constant__ AngTab T, double* __restrict__ ang) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= npairs) return;
  const FarPair p = pairs[k];
  const DropDev Di = drops[p.i], Dj = drops[p.j];
  const double tx = Di.cx - Dj.cx, ty = Di.cy - Dj.cy, tz = Di.cz - Dj.cz;
  const double h2 = tx * tx + ty * ty, h = sqrt(h2), iD = 1.0 / sqrt(h2 + tz * tz);
  const double cp = h > 0.0 ? tx / h : 1.0, sp = h > 0.0 ? ty / h : 0.0, ct = tz * iD, st = h * iD;
  const double gs = 2.0 * iD / (double)inv_src[p.j], gt = 2.0 * iD / (double)inv_tgt[p.i];
  double* a = ang + p.ang;
  const int n1 = p.L + 1;
  double c1 = 1.0, s1 = 0.0, c2 = 1.0, s2 = 0.0, ps = 12.566370614359172954, pt = iD;
  for (int m = 0; m < n1; ++m) {
    a[m] = c1;
    a[n1 + m] = s1;
    a[2 * n1 + m] = c2;
    a[3 * n1 + m] = s2;
    a[4 * n1 + m] = T.r[m] * ps;
    a[5 * n1 + m] = T.r[m] * pt;
    const double u = c1 * cp - s1 * sp, v = c2 * ct - s2 * st;
    s1 = c1 * sp + s1 * cp;
    s2 = c2 * st + s2 * ct;
    c1 = u;
    c2 = v;
    ps *= gs;
    pt *= gt;
  }
}

// order at which the targets of a group may take the expansion of an entry's drop: a warp per group
__global__ void k_far_reach(int nent, const int* __restrict__ ent_tgt, NearList nl, int64_t ngroup,
                            const DropDev* __restrict__ drops, const unsigned* __restrict__ ext,
                            const int* __restrict__ Lsrc, const __grid_constant__ RhoReach R,
                            const double* __restrict__ tgt, int64_t ntarget, unsigned char* __restrict__ order) {
  const int64_t f = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (f >= ngroup) return;
  const int en = entry_of(nl.goff, nent, f), lane = threadIdx.x & 31;
  const int j = nl.drop[en];
  const DropDev Di = drops[ent_tgt[en]], Dj = drops[j];
  const int64_t sl = (f - nl.goff[en]) * kFarGroup + lane;
  double d2 = INFINITY;
  if (sl < Di.nt) {
    const int64_t t = nl.tgt[Di.tgt_off + sl];
    const double dx = tgt[t] - Dj.cx, dy = tgt[ntarget + t] - Dj.cy, dz = tgt[2 * ntarget + t] - Dj.cz;
    d2 = dx * dx + dy * dy + dz * dz;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d2 = fmin(d2, __shfl_xor_sync(0xffffffffu, d2, o));
  if (lane) return;
  const float rho = (float)((double)__uint_as_float(ext[j]) / sqrt(d2)) * 1.000001f;
  int L = 2;
  while (L <= Lsrc[j] && !(rho <= R.r[L])) ++L;
  order[f] = (unsigned char)(L <= Lsrc[j] ? L : kNoReach);
}

// every other drop, in the order of the layout
__global__ void k_far_all(const DropDev* __restrict__ drops, int nd, int64_t nsource, int64_t* __restrict__ pre,
                          int* __restrict__ drop, unsigned* __restrict__ off) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
  if (e >= nd) return;
  const bool end = e == nd - 1;
  const int j = e + (e >= i ? 1 : 0);
  const int64_t at = (int64_t)i * nd + e, before = end ? nsource : drops[j].src_off;
  drop[at] = end ? -1 : j;
  pre[at] = before - (end || j > i ? (int64_t)drops[i].ns : 0);
  if (e == 0) off[i] = (unsigned)i * (unsigned)nd;
  if (end && i == nd - 1) off[nd] = (unsigned)nd * (unsigned)nd;
}

// target-source pairs of the groups that are summed directly
__global__ void k_far_direct(int nent, const int* __restrict__ ent_tgt, NearList nl, int64_t ngroup,
                             const DropDev* __restrict__ drops, double* __restrict__ sum) {
  double n = 0.0;
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < ngroup; f += (int64_t)gridDim.x * blockDim.x) {
    const int en = entry_of(nl.goff, nent, f), g = (int)(f - nl.goff[en]);
    const int ns = drops[nl.drop[en]].ns, nt = drops[ent_tgt[en]].nt;
    if (nl.direct(en, g, ns)) n += (double)ns * min(kFarGroup, nt - g * kFarGroup);
  }
  n = warp_add(n);
  if ((threadIdx.x & 31) == 0 && n != 0.0) atomicAdd(sum, n);   // whole numbers: exact in any order
}

// FP32 instructions of a direct pair and of the expansions' inner steps (double-float 12 per multiply-add, FP64 64
// issue slots per instruction), by kind DL, SL, S + D, S, D
constexpr double kDirect32[5] = {25.0, 18.0, 45.0, 35.0, 37.0};
constexpr double kDirectDf[5] = {121.0, 78.0, 260.0, 187.0, 195.0};
constexpr double kDirect64[5] = {1060.0, 740.0, 1980.0, 1540.0, 1470.0};

}  // namespace

void far_release(shbim_ctx* ctx) {
  FarState& F = *ctx->far;
  auto drop = [](auto*& p, size_t& cap) {
    cudaFree(p);
    p = nullptr;
    cap = 0;
  };
  drop(F.blob, F.blob_cap);
  drop(F.lists, F.lists_cap);
  drop(F.ang, F.ang_cap);
  drop(F.q, F.q_cap);
  drop(F.part, F.part_cap);
  drop(F.v, F.v_cap);
  drop(F.mom, F.mom_cap);
  drop(F.lpair, F.lpair_cap);
  drop(F.loc, F.loc_cap);
  drop(F.set, F.set_cap);
  drop(F.mset, F.mset_cap);
  drop(F.order, F.order_cap);
  drop(F.mpart, F.mpart_cap);
}

void far_free(shbim_ctx* ctx) {
  if (!ctx->far) return;
  FarState& F = *ctx->far;
  far_release(ctx);
  cudaFree(F.tables);
  cudaFree(F.all);
  cudaFree(F.count);
  cudaFreeHost(F.count_host);
  delete ctx->far;
  ctx->far = nullptr;
}

void far_forget(shbim_ctx* ctx, bool layout) {
  if (!ctx->far) return;
  if (layout) ctx->far->all_drops = 0;
  for (auto& P : ctx->far->plan) P = FarPlan{};
}

int far_count(shbim_ctx* ctx, cudaStream_t s) {
  if (!ctx->far) ctx->far = new FarState();
  FarState& F = *ctx->far;
  const size_t n = (size_t)kFarPlans * ctx->n_drops;
  const size_t lsrc_off = (size_t)kFarRows * ctx->n_drops * sizeof(FarRow), sum_off = (lsrc_off + n * sizeof(int) + 15) / 16 * 16;
  if (int rc = far_grow(ctx, (void**)&F.count, &F.count_cap, sum_off + sizeof(double), "drop pair counts")) return rc;
  if (F.count_host_cap < sum_off) {
    cudaFreeHost(F.count_host);
    F.count_host = nullptr;
    F.count_host_cap = 0;
    if (cudaMallocHost((void**)&F.count_host, sum_off) != cudaSuccess) {
      cudaGetLastError();
      return fail(ctx, SHBIM_ERR_NOMEM, "cudaMallocHost drop pair counts");
    }
    F.count_host_cap = sum_off;
  }
  F.sum = reinterpret_cast<double*>(F.count + sum_off);
  FarRow* rows = reinterpret_cast<FarRow*>(F.count);
  int* lsrc = reinterpret_cast<int*>(F.count + lsrc_off);
  SHBIM_CUDA(ctx, cudaMemsetAsync(lsrc, 0xff, n * sizeof(int), s));   // -1
  k_far_count<<<(unsigned)((ctx->n_drops * 32 + 127) / 128), 128, 0, s>>>(rho_tab(), ctx->centres_dev, ctx->dq_ext_dev,
                                                                         ctx->drops_dev, ctx->n_drops, rows, lsrc);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_count");
  SHBIM_CUDA(ctx, cudaMemcpyAsync(F.count_host, F.count, sum_off, cudaMemcpyDeviceToHost, s));
  return SHBIM_OK;
}

// Plans in use: their per-drop lists (uploaded), per-pair lists (k_far_fill) and the workspaces of their expansions.
int build_far(shbim_ctx* ctx, const std::vector<double>& ext, cudaStream_t s) {
  FarState& F = *ctx->far;
  const int nd = ctx->n_drops;
  std::vector<unsigned char> blob;
  auto put = [&](const void* p, size_t bytes) {
    const size_t o = (blob.size() + 15) / 16 * 16;
    blob.resize(o + bytes);
    if (bytes) std::memcpy(blob.data() + o, p, bytes);
    return o;
  };
  size_t lists = 0;
  auto room = [&](size_t bytes) {
    const size_t o = lists;
    lists = (o + bytes + 15) / 16 * 16;
    return o;
  };
  struct Offsets {
    size_t off, lsrc, sd, td, chunks, blocks, pairs, drop, ent_tgt, pre, goff;
  } off[kFarPlans] = {};
  size_t all_off = 0;                          // every pair with angles
  double cross = 0.0;
  for (const Drop& d : ctx->drops) cross += (double)d.nt * (double)(ctx->nsource - d.ns);
  // every other drop: once per layout
  const size_t n2 = (size_t)nd * nd;
  if (F.all_drops != nd) {
    if (int rc = far_grow(ctx, (void**)&F.all, &F.all_cap, n2 * (sizeof(int64_t) + sizeof(int)) + (nd + 1) * sizeof(unsigned),
                          "list of all drop pairs"))
      return rc;
    k_far_all<<<dim3((unsigned)((nd + 127) / 128), (unsigned)nd), 128, 0, s>>>(
        ctx->drops_dev, nd, ctx->nsource, reinterpret_cast<int64_t*>(F.all), reinterpret_cast<int*>(F.all + n2 * sizeof(int64_t)),
        reinterpret_cast<unsigned*>(F.all + n2 * (sizeof(int64_t) + sizeof(int))));
    SHBIM_CHECK_LAUNCH(ctx, "k_far_all");
    F.all_drops = nd;
  }
  NearList& others = F.plan[kFarPlans].near;
  others.pre = reinterpret_cast<const int64_t*>(F.all);
  others.drop = reinterpret_cast<const int*>(F.all + n2 * sizeof(int64_t));
  others.off = reinterpret_cast<const unsigned*>(F.all + n2 * (sizeof(int64_t) + sizeof(int)));
  others.tgt = ctx->tgt_order;
  F.plan[kFarPlans].direct_pairs = cross;
  std::vector<float> inv(2 * nd, 1.f);
  for (int i = 0; i < 2 * nd; ++i) {
    int e = 0;
    std::frexp(ext[i], &e);                 // ext < 2^e
    inv[i] = (float)std::ldexp(1.0, -e);
  }
  const size_t inv_off = put(inv.data(), inv.size() * sizeof(float));
  size_t max_part = 0, max_v = 0, max_mom = 0, max_lp = 0, max_loc = 0, max_set = 0, max_mset = 0, max_mpart = 0;
  size_t group_total = 0;
  const FarRow* all = reinterpret_cast<const FarRow*>(F.count_host) + (size_t)kFarPlans * nd;
  int64_t all_pairs = 0, ang_total = 0;
  for (int i = 0; i < nd; ++i) {
    all_pairs += all[i].far;
    ang_total += all[i].ang;
  }
  if (all_pairs > INT32_MAX) return SHBIM_OK;
  int max_charges = 0;
  bool used[kFarPlans] = {};
  for (int pl = 0; pl < kFarPlans; ++pl) {
    FarPlan& P = F.plan[pl];
    const FarRow* row = reinterpret_cast<const FarRow*>(F.count_host) + (size_t)pl * nd;
    const int* Lsrc = reinterpret_cast<const int*>(F.count_host + (size_t)kFarRows * nd * sizeof(FarRow)) + (size_t)pl * nd;
    int64_t npairs = 0, nent = 0;
    for (int i = 0; i < nd; ++i) {
      npairs += row[i].far;
      nent += nd - row[i].far;                // the others and the end of the list
      P.far_pairs += (double)row[i].pairs;
      const int nt = ctx->drops[i].nt;
      P.far_warps += (double)row[i].pairs / nt * ((nt + 31) / 32 * 32);
      P.far_ctas += (double)row[i].pairs * std::min(2.5, (double)((nt + 127) / 128 * 128) / nt);
      P.pair_work += row[i].cubes;
      P.lmax = std::max(P.lmax, row[i].lmax);
      P.tgt_work += (double)ctx->drops[i].nt * (row[i].lmax < 0 ? 0 : FarReach::tri(row[i].lmax));
      P.src_work += (double)ctx->drops[i].ns * (Lsrc[i] < 0 ? 0 : FarReach::tri(Lsrc[i]));
    }
    P.direct_pairs = cross - P.far_pairs;
    if (npairs == 0 || npairs > INT32_MAX || nent > INT32_MAX) continue;
    P.npairs = (int)npairs;
    P.nent = (int)nent;
    // which kinds are worth it
    for (int k = 0; k < 5; ++k) {
      P.use[k] = kDerivs[k] == pl % 3 && far_worth(P, pl / 3, k);
      used[pl] = used[pl] || P.use[k];
    }
    if (!used[pl]) continue;
    std::vector<unsigned> nb_off(nd + 1, 0);
    std::vector<FarSrcDrop> sd(nd);
    std::vector<FarTgtDrop> td(nd);
    std::vector<FarChunk> chunks;
    std::vector<int2> blocks;
    int pair = 0;
    int64_t ang = 0;
    for (int i = 0; i < nd; ++i) {
      const Drop& d = ctx->drops[i];
      const int near = nd - 1 - row[i].far;
      nb_off[i + 1] = nb_off[i] + near + 1;
      td[i] = FarTgtDrop{row[i].lmax, pair, pair + row[i].far, P.loc, P.tri, P.lout, ang, P.ngroup};
      if (P.batches.empty() || P.lout + row[i].out - P.batches.back().out0 > kFarBatch)
        P.batches.push_back(FarBatch{i, i, pair, pair, P.lout, P.lout});
      pair += row[i].far;
      P.lout += row[i].out;
      P.batches.back().drop1 = i + 1;
      P.batches.back().pair1 = pair;
      P.batches.back().out1 = P.lout;
      ang += all[i].ang;
      P.ngroup += (int64_t)near * ((d.nt + kFarGroup - 1) / kFarGroup);
      if (row[i].lmax >= 0) {
        P.loc += (int64_t)(row[i].lmax + 1) * (row[i].lmax + 1);
        P.tri += FarReach::tri(row[i].lmax);
        for (int t = 0; t < d.nt; t += 32) blocks.push_back(make_int2(i, t));
      }
      sd[i] = FarSrcDrop{P.part, P.coef, P.stri, 0};
      if (Lsrc[i] < 0) continue;
      for (int f = 0; f < d.ns; f += kP2mSrc) {
        chunks.push_back(FarChunk{i, f, std::min(kP2mSrc, d.ns - f), 0, P.part});
        P.part += FarReach::tri(Lsrc[i]);
        sd[i].nchunk++;
      }
      P.coef += (int64_t)(Lsrc[i] + 1) * (Lsrc[i] + 1);
      P.stri += FarReach::tri(Lsrc[i]);
    }
    P.nchunks = (int)chunks.size();
    P.nblocks = (int)blocks.size();
      for (int k = 0; k < 5; ++k) {
        if (!P.use[k]) continue;
        const size_t npot = stokes_like(k) ? 4 : 1;
        max_part = std::max(max_part, (size_t)2 * kCharges[k] * P.part);
        max_v = std::max(max_v, (size_t)kCharges[k] * P.coef);
        if (k == 2 || k == 4) max_mom = std::max(max_mom, (size_t)4 * P.coef);
        for (const FarBatch& b : P.batches) max_lp = std::max(max_lp, npot * (size_t)(b.out1 - b.out0));
        max_loc = std::max(max_loc, npot * (size_t)P.loc);
        max_set = std::max(max_set, (size_t)2 * kSets[k] * P.tri);
        max_mset = std::max(max_mset, (size_t)2 * kSets[k] * P.stri);
        max_mpart = std::max(max_mpart, (size_t)(stokes_like(k) ? 96 : 32) * P.ngroup);
        max_charges = std::max(max_charges, kCharges[k]);
      }
    group_total += (size_t)P.ngroup;
    Offsets& o = off[pl];
    o.off = put(nb_off.data(), nb_off.size() * sizeof(unsigned));
    o.lsrc = put(Lsrc, nd * sizeof(int));
    o.sd = put(sd.data(), sd.size() * sizeof(FarSrcDrop));
    o.td = put(td.data(), td.size() * sizeof(FarTgtDrop));
    o.chunks = put(chunks.data(), chunks.size() * sizeof(FarChunk));
    o.blocks = put(blocks.data(), blocks.size() * sizeof(int2));
    o.pairs = room((size_t)npairs * sizeof(FarPair));
    o.drop = room((size_t)nent * sizeof(int));
    o.ent_tgt = room((size_t)nent * sizeof(int));
    o.pre = room((size_t)nent * sizeof(int64_t));
    o.goff = room((size_t)(nent + 1) * sizeof(int64_t));
  }
  if (std::none_of(used, used + kFarPlans, [](bool u) { return u; })) return SHBIM_OK;
  // where a drop's pairs with angles start
  size_t all_td;
  {
    std::vector<FarTgtDrop> td(nd);
    int pair = 0;
    int64_t ang = 0;
    for (int i = 0; i < nd; ++i) {
      td[i] = FarTgtDrop{-1, pair, pair + all[i].far, 0, 0, 0, ang, 0};
      pair += all[i].far;
      ang += all[i].ang;
    }
    all_td = put(td.data(), td.size() * sizeof(FarTgtDrop));
    all_off = room((size_t)all_pairs * sizeof(FarPair));
  }
  // The expansions take at most half of the memory that is free: near grids, the row build's lanes and the solvers'
  // vectors come after them. Where that, or an allocation, falls short, they give everything back and every pair is
  // summed directly.
  struct Want {
    void** p;
    size_t* cap;
    size_t bytes;
    const char* what;
  };
  const Want want[] = {{(void**)&F.blob, &F.blob_cap, blob.size(), "expansion plans"},
                       {(void**)&F.lists, &F.lists_cap, lists, "drop pair lists"},
                       {(void**)&F.ang, &F.ang_cap, (size_t)ang_total * 8, "expansion angles"},
                       {&F.q, &F.q_cap, (size_t)max_charges * ctx->nsource * 8, "expansion charges"},
                       {&F.part, &F.part_cap, max_part * 8, "expansion partial moments"},
                       {&F.v, &F.v_cap, max_v * 8, "expansion moments"},
                       {&F.mom, &F.mom_cap, max_mom * 8, "expansion dipole moments"},
                       {&F.lpair, &F.lpair_cap, max_lp * 8, "expansion pair terms"},
                       {&F.loc, &F.loc_cap, max_loc * 8, "local expansions"},
                       {&F.set, &F.set_cap, max_set * 8, "local expansions of derivatives"},
                       {&F.order, &F.order_cap, std::max<size_t>(group_total, 1), "orders of close pairs"},
                       {&F.mset, &F.mset_cap, max_mset * 8, "multipole expansions of derivatives"},
                       {&F.mpart, &F.mpart_cap, max_mpart * 8, "values of multipole expansions"}};
  size_t more = 0, held = 0;
  for (const Want& w : want) {
    held += *w.cap;
    more += w.bytes > *w.cap ? w.bytes : 0;
  }
  int rc = SHBIM_OK;
  if (more > 0) {
    size_t free_bytes = 0, total = 0;
    SHBIM_CUDA(ctx, cudaMemGetInfo(&free_bytes, &total));
    if (more > (free_bytes + held) / 2) rc = SHBIM_ERR_NOMEM;
  }
  if (!rc) rc = far_tables(ctx);
  for (const Want& w : want)
    if (!rc) rc = far_grow(ctx, w.p, w.cap, w.bytes, w.what);
  if (rc == SHBIM_ERR_NOMEM) {
    far_release(ctx);
    for (int pl = 0; pl < kFarPlans; ++pl) F.plan[pl] = FarPlan{};
    ctx->err.clear();
    return SHBIM_OK;
  }
  if (rc) return rc;
  SHBIM_CUDA(ctx, cudaMemcpyAsync(F.blob, blob.data(), blob.size(), cudaMemcpyHostToDevice, s));
  SHBIM_CUDA(ctx, cudaStreamSynchronize(s));   // the host copy goes away
  F.inv_src = reinterpret_cast<const float*>(F.blob + inv_off);
  F.inv_tgt = F.inv_src + nd;
  FillPlans fill{};
  int nfill = 0;
  size_t go = 0;
  for (int pl = 0; pl < kFarPlans; ++pl) {
    if (!used[pl]) continue;
    FarPlan& P = F.plan[pl];
    const Offsets& o = off[pl];
    P.near = F.plan[kFarPlans].near;
    P.near.off = reinterpret_cast<const unsigned*>(F.blob + o.off);
    P.near.drop = reinterpret_cast<const int*>(F.lists + o.drop);
    P.near.pre = reinterpret_cast<const int64_t*>(F.lists + o.pre);
    P.near.goff = reinterpret_cast<const int64_t*>(F.lists + o.goff);
    P.ent_tgt = reinterpret_cast<const int*>(F.lists + o.ent_tgt);
    P.pairs = reinterpret_cast<const FarPair*>(F.lists + o.pairs);
    P.Lsrc = reinterpret_cast<const int*>(F.blob + o.lsrc);
    P.sd = reinterpret_cast<const FarSrcDrop*>(F.blob + o.sd);
    P.td = reinterpret_cast<const FarTgtDrop*>(F.blob + o.td);
    P.chunks = reinterpret_cast<const FarChunk*>(F.blob + o.chunks);
    P.blocks = reinterpret_cast<const int2*>(F.blob + o.blocks);
    P.order = static_cast<unsigned char*>(F.order) + go;
    go += (size_t)P.ngroup;
    fill.p[nfill++] = FillPlan{pl, P.td, P.near.off, const_cast<FarPair*>(P.pairs), const_cast<int*>(P.near.drop),
                               const_cast<int*>(P.ent_tgt), const_cast<int64_t*>(P.near.pre),
                               const_cast<int64_t*>(P.near.goff)};
  }
  FarPair* all_dev = reinterpret_cast<FarPair*>(F.lists + all_off);
  fill.p[nfill++] = FillPlan{kFarPlans, reinterpret_cast<const FarTgtDrop*>(F.blob + all_td), nullptr, all_dev,
                             nullptr, nullptr, nullptr, nullptr};
  k_far_fill<<<dim3((unsigned)((nd * 32 + 127) / 128), (unsigned)nfill), 128, 0, s>>>(
      rho_tab(), fill, ctx->centres_dev, ctx->dq_ext_dev, ctx->drops_dev, nd);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_fill");
  AngTab A;
  for (int m = 0; m <= kFarCapMax; ++m) A.r[m] = 1.0 / std::sqrt(2.0 * m + 1.0);
  k_far_angles<<<(unsigned)((all_pairs + 63) / 64), 64, 0, s>>>(all_dev, (int)all_pairs, ctx->drops_dev, F.inv_src, F.inv_tgt,
                                                              A, F.ang);
  SHBIM_CHECK_LAUNCH(ctx, "k_far_angles");
  for (int pl = 0; pl < kFarPlans; ++pl) {
    if (!used[pl]) continue;
    FarPlan& P = F.plan[pl];
    if (P.ngroup == 0) continue;
    RhoReach R{};
    for (int L = 0; L <= plan_cap(pl); ++L) R.r[L] = std::nextafterf((float)rho_tab().r[pl][L], 0.f);
    k_far_reach<<<(unsigned)((P.ngroup * 32 + 255) / 256), 256, 0, s>>>(
        P.nent, P.ent_tgt, P.near, P.ngroup, ctx->drops_dev, ctx->dq_ext_dev, P.Lsrc, R, ctx->geo.tgt, ctx->ntarget, P.order);
    SHBIM_CHECK_LAUNCH(ctx, "k_far_reach");
    P.near.order = P.order;
  }
  return SHBIM_OK;
}

// What the expansions of a plan cost against the direct sums they replace, in FP32 instructions of the whole GPU (37 per
// ns): their inner steps, half as much again for latency and reads (twice in FP64); a term per pair of drops and potential
// for the short loops and barriers of k_far_m2l and k_far_lsum (8 to 10 ns in FP32 sums and 19 to 22 in double-float
// at 1024 drops, inner steps included); the launches and the chain of dependent kernels, 80 to 220 us. A direct sum pays
// for whole warps of targets (FP32) or whole CTAs of 128, of which at most 2.5 lanes per target were seen to count.
// Both sides were measured on lattices of 6 to 1024 drops of degree 3 to 24, every kind and precision: the rule picks
// the faster one beyond 10 % of its crossings but for a few sums of drops of degree 3. Without the term per pair, FP32
// Stokes sums took the expansions for 1024 drops of degree 4 (40.4 ms, 15.8 directly) and 128 of degree 6 (1.31, 0.84).
// 64 drops of degree 8, double layer, with expansions and directly: FP32 0.31 and 0.46 ms, double-float 0.86 and 2.40,
// FP64 3.8 and 27.5. 16 drops of degree 11, Stokeslet in double-float: 0.63 and 0.56 ms, left direct. Solves of eight
// FP64 applications to six drops of degree 16 in boxes lie at the crossing: 12.0 to 14.4 ms where the rule takes the
// expansions, 14.0 to 14.9 directly.
bool far_worth(const FarPlan& P, int precision, int kind) {
  const bool fp64 = precision == SHBIM_PREC_FP64, fp32 = precision == SHBIM_PREC_FP32_COMP;
  const double* direct = fp32 ? kDirect32 : (fp64 ? kDirect64 : kDirectDf);
  const int npot = stokes_like(kind) ? 4 : 1;
  const double inner = P.src_work * (45.0 + 26.0 * kCharges[kind]) + P.tgt_work * (30.0 + 26.0 * kSets[kind]) +
                       P.pair_work * npot * 30.0;
  const double unit = fp64 ? 2.0 * 64.0 / 12.0 : 1.5, pair = fp32 ? (npot == 1 ? 2e5 : 3.2e5) : (fp64 ? 1.1e6 : 4.5e5);
  const double launches = npot == 1 ? (fp32 ? 3e9 : 5e9) : (fp32 ? 5.5e9 : 8e9);
  return P.npairs > 0 &&
         unit * inner + pair * npot * P.npairs + launches < (fp32 ? P.far_warps : P.far_ctas) * direct[kind];
}

const FarPlan* far_plan(const shbim_ctx* ctx, int kind) {
  if (!ctx->far || !ctx->expansions) return nullptr;
  const FarPlan& P = ctx->far->plan[3 * ctx->opts.precision + kDerivs[kind]];
  return P.use[kind] ? &P : nullptr;
}

const FarPlan& far_all(const shbim_ctx* ctx) { return ctx->far->plan[kFarPlans]; }

bool far_ready(const shbim_ctx* ctx) { return ctx->n_drops < 2 || (ctx->far && far_all(ctx).near.tgt); }

// Instructions of an expansion's value: recurrence and 2 NS multiply-adds per (n, m), half as much again for reads
// and orders of uneven length; `base` for the powers of x + iy and the sums over warps. In FP64 four times that: six
// drops of degree 16, double layer, solve of eight applications: 16.9 ms without these expansions, 16.3 at one
// time, 15.7 at four. 64 drops of degree 16 to 48, without and with them: Stokeslet in double-float 35.5 and 24.2 ms,
// stresslet FP32 10.2 and 9.0, double layer FP32 3.83 and 2.88; twice the instructions here change nothing. Below 0.1 ms
// of direct sums the three launches cost more than they give (40 drops of degree 11, 3e9: 1.00 and 1.03 ms).
NearList far_near(const shbim_ctx* ctx, const FarPlan& P, int kind) {
  NearList nl = P.near;
  const int ns = kSets[kind], pr = ctx->opts.precision;
  const double direct = (pr == SHBIM_PREC_FP64 ? kDirect64 : (pr == SHBIM_PREC_DF64 ? kDirectDf : kDirect32))[kind];
  if (P.direct_pairs * direct < 4e9) nl.order = nullptr;
  FarReach& r = nl.reach;
  if (pr == SHBIM_PREC_FP64) {
    r = FarReach{kFarLmax, 384 * (3 + 2 * ns), 0, 120000, (int)direct};
  } else {
    const bool fp32 = pr == SHBIM_PREC_FP32_COMP;
    r = FarReach{fp32 ? 12 : 36, 50 + 36 * ns, 9 + 6 * ns, 15000, (int)direct};
  }
  return nl;
}

double far_direct_pairs(const shbim_ctx* ctx, const FarPlan& P, int kind) {
  if (P.counted[kind]) return P.count[kind];
  const NearList nl = far_near(ctx, P, kind);
  if (!nl.order) return P.direct_pairs;
  double n = 0.0;
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemset(ctx->far->sum, 0, sizeof(double)) != cudaSuccess) return P.direct_pairs;
  k_far_direct<<<(unsigned)std::min<int64_t>((P.ngroup + 255) / 256, 1024), 256>>>(P.nent, P.ent_tgt, nl, P.ngroup,
                                                                                  ctx->drops_dev, ctx->far->sum);
  if (cudaMemcpy(&n, ctx->far->sum, sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    return P.direct_pairs;
  }
  P.counted[kind] = true;
  return P.count[kind] = n;
}

}  // namespace shbim
