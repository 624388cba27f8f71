// Plans (far_plan.cu) and workspaces of the expansions between well-separated drops (far.cu).
#pragma once

#include <cstdint>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"

namespace shbim {

constexpr int kFarLmax = 63;        // orders the constant tables hold
// Levels of truncation by precision (FP64, FP32, double-float: the order of SHBIM_PREC_*): bound of a pair's error
// relative to strengths over gap, and largest order of a far pair. What they come to is below the rounding of the direct
// sums, 7e-16 to 2e-15 of a target's sum of magnitudes in FP64, 1e-12 in double-float, 1e-7 in FP32; FP64 sums take one
// order more up to kFarTight, where the sources of a distant drop lie in one direction and the bound is nearly reached:
// 57 radii away the double layer was 1.4e-15 off without it, 8.8e-16 summed directly. One bound of 1e-15 for every pair
// made solves of six drops of degree 16 3 % slower: the order of the closest pair sets the time of k_far_m2l there.
constexpr double kFarEps[3] = {3e-15, 1e-8, 3e-15};
constexpr int kFarTight = 24;
__host__ __device__ constexpr int far_cap(int precision) { return precision == 1 ? 36 : 60; }
constexpr int kFarPlans = 9;        // [precision][derivatives]
constexpr int kFarCapMax = 60;
static_assert(kFarCapMax <= kFarLmax, "the tables hold every order");
constexpr int kP2mSrc = 1024;       // sources of a chunk of the moments (a CTA of k_far_p2m)
// by kind (0 DL, 1 SL, 2 S + D, 3 S, 4 D): expansions the targets evaluate, charges of a source, derivatives taken of
// 1/r in the truncation bound
constexpr int kSets[5] = {3, 1, 12, 12, 12};
constexpr int kCharges[5] = {1, 1, 13, 4, 9};
constexpr int kDerivs[5] = {1, 0, 2, 1, 2};

// charge sets of the moments: Laplace strengths; f, y.f; dipole tensor and vector; both
enum FarMode { kFarLap = 0, kFarS = 1, kFarD = 2, kFarSD = 3 };

inline bool stokes_like(int kind) { return kind >= 2; }

struct FarPair {
  int i, j, L;
  int na;             // rows of its angles and powers, six of them (they serve every plan)
  int64_t out;        // offset of the pair's local terms (coefficients, per potential)
  int64_t ang;        // offset of its angles and powers
};
struct FarChunk {
  int drop, first, count, pad;
  int64_t part;       // offset of its partial moments (in units of tri(L))
};
struct FarSrcDrop {
  int64_t part, coef, tri;
  int nchunk;
};
struct FarTgtDrop {
  int L, pair0, pair1;
  int64_t coef, tri;
  int64_t out, ang, group;            // where its pairs' local terms and angles and its entries' groups start
};

// What a target's value of a multipole expansion of order L costs against the direct sum over ns sources, in
// instructions: `full` per (n, m) of degrees up to nf, `low` above, `base` per expansion, `direct` per source.
// Whole numbers, so that every kernel that asks comes to the same answer.
struct FarReach {
  int nf = 0, full = 0, low = 0, base = 0, direct = 0;
  __host__ __device__ static int tri(int L) { return (L + 1) * (L + 2) / 2; }
  __host__ __device__ bool worth(int L, int ns) const {
    const int k = tri(L < nf ? L : nf);
    return (int64_t)full * k + (int64_t)low * (tri(L) - k) + base < (int64_t)direct * ns;
  }
};

constexpr int kFarGroup = 32;       // targets that share a decision
constexpr int kNoReach = 255;

// Per target drop i the drops that no local expansion covers (or all others), entries [off[i], off[i+1]): drop index and
// the number of sources before it in the list; the last entry of a drop has index -1 and the total. The targets of a drop
// are taken in the order tgt[] (patches of the surface); group g of 32 of them reaches the multipole expansion of the
// entry's drop at order order[goff[entry] + g] (kNoReach: at none), and is summed directly where that is not worth it.
// Entries are unsigned: the list of all others holds the square of up to 65535 drops.
struct NearList {
  const unsigned* off = nullptr;
  const int* drop = nullptr;
  const int64_t* pre = nullptr;
  const int* tgt = nullptr;
  const int64_t* goff = nullptr;    // [entries + 1]
  const unsigned char* order = nullptr;   // null: every group directly
  FarReach reach;
  __host__ __device__ bool direct(unsigned entry, int group, int ns) const {
    if (!order) return true;
    const int L = order[goff[entry] + group];
    return L == kNoReach || !reach.worth(L, ns);
  }
};

// the entry whose groups hold flat group f
__device__ __forceinline__ int entry_of(const int64_t* __restrict__ goff, int nent, int64_t f) {
  int a = 0, b = nent;                    // goff[a] <= f < goff[b]
  while (b - a > 1) {
    const int c = (a + b) >> 1;
    if (goff[c] <= f)
      a = c;
    else
      b = c;
  }
  return a;
}

template <class T>
struct FarTab {
  const T *dq_r, *dq_c, *tr, *kap, *rec, *la, *lp, *lq;
  const int *dq_off, *tr_off;
  const int2 *pat_r, *pat_c;
};

// target drops whose pair terms are held at once: their pairs and the terms' place
struct FarBatch {
  int drop0, drop1, pair0, pair1;
  int64_t out0, out1;
};
constexpr int64_t kFarBatch = int64_t(1) << 26;   // coefficients per potential (2 GB for the four of a Stokes sum)

struct FarPlan {
  NearList near;
  double direct_pairs = 0.0, far_pairs = 0.0;
  double far_warps = 0.0, far_ctas = 0.0;   // far pairs with the targets of a drop rounded up to warps, to 128
  double src_work = 0.0, tgt_work = 0.0, pair_work = 0.0;
  int npairs = 0, nchunks = 0, nblocks = 0, lmax = 0;
  int64_t part = 0, coef = 0, loc = 0, lout = 0, tri = 0;
  bool use[5] = {};                   // [kind]
  const FarPair* pairs = nullptr;
  const int* Lsrc = nullptr;
  const FarSrcDrop* sd = nullptr;
  const FarTgtDrop* td = nullptr;
  const FarChunk* chunks = nullptr;
  const int2* blocks = nullptr;
  // close pairs: groups of targets far enough for the source drop's own expansion
  int nent = 0;
  int64_t ngroup = 0, stri = 0;
  const int* ent_tgt = nullptr;       // target drop of an entry (-1: end of a list)
  unsigned char* order = nullptr;     // [ngroup]
  std::vector<FarBatch> batches;
  // pairs summed directly, by kind, once they have been asked for
  mutable bool counted[5] = {};
  mutable double count[5] = {};
};

// What a target drop's row of the drop pairs comes to under one plan, or (the last row) where a pair has the largest
// order that any plan gives it (k_far_count)
struct FarRow {
  int64_t out;                        // sum of (L + 1)^2 over its far drops
  int64_t pairs;                      // targets times sources of its far drops
  double cubes;                       // sum of 2 L^3
  int far, lmax, ang, pad;            // far drops, largest order, sum of 6 (L + 1)
};
constexpr int kFarRows = kFarPlans + 1;

struct FarState {
  FarPlan plan[kFarPlans + 1];        // the last one: every other drop directly
  unsigned char* blob = nullptr;      // per-drop lists of the plans in use, written by the host
  size_t blob_cap = 0;
  unsigned char* lists = nullptr;     // per-pair lists of the plans in use, written by k_far_fill
  size_t lists_cap = 0;
  unsigned char* all = nullptr;       // list of all others: [n_drops^2] int64 and int, [n_drops + 1] offsets
  size_t all_cap = 0;
  int all_drops = 0;                  // drops of the layout it was made for (0: none)
  unsigned char* count = nullptr;     // [kFarRows][n_drops] FarRow, [kFarPlans][n_drops] largest order of a source drop, a sum
  unsigned char* count_host = nullptr;   // page-locked, the same
  size_t count_cap = 0, count_host_cap = 0;
  double* sum = nullptr;              // in count: pairs summed directly, when asked for
  void* tables = nullptr;
  FarTab<double> td{};
  FarTab<dfl::df> tf{};
  const float* inv_src = nullptr;     // per drop 1 / A (sources) and 1 / B (targets), powers of two
  const float* inv_tgt = nullptr;
  double* ang = nullptr;
  size_t ang_cap = 0;
  void *q = nullptr, *part = nullptr, *v = nullptr, *mom = nullptr, *lpair = nullptr, *loc = nullptr, *set = nullptr;
  size_t q_cap = 0, part_cap = 0, v_cap = 0, mom_cap = 0, lpair_cap = 0, loc_cap = 0, set_cap = 0;
  void *mset = nullptr, *order = nullptr, *mpart = nullptr;
  size_t mset_cap = 0, order_cap = 0, mpart_cap = 0;
};

// Lists of direct and far drop pairs of the current geometry. far_count queues the classification of all pairs under
// every plan behind the extents (ctx->dq_ext_dev) and their read-back; after a synchronisation build_far decides which
// plans are used and makes their lists, ext holding per drop the largest |x - c| of the sources, then of the targets.
int far_count(shbim_ctx* ctx, cudaStream_t s);
int build_far(shbim_ctx* ctx, const std::vector<double>& ext, cudaStream_t s);
// expansion tables on the device (far.cu)
int far_tables(shbim_ctx* ctx);
int far_grow(shbim_ctx* ctx, void** p, size_t* cap, size_t bytes, const char* what);
void far_free(shbim_ctx* ctx);
// gives the lists and workspaces back
void far_release(shbim_ctx* ctx);
// empties every plan (the workspaces stay): what comes before build_far may fail; with the layout the list of all
// others too
void far_forget(shbim_ctx* ctx, bool layout = false);
// whether the expansions pay for this kind of sum at this precision
bool far_worth(const FarPlan& P, int precision, int kind);
// the plan of a kind (0 DL, 1 SL, 2 S + D, 3 S, 4 D) at the context's precision, null: all pairs directly
const FarPlan* far_plan(const shbim_ctx* ctx, int kind);
const FarPlan& far_all(const shbim_ctx* ctx);
// the lists of the current shapes have been made (or none are needed)
bool far_ready(const shbim_ctx* ctx);
// the plan's lists with the rule of a kind at the context's precision
NearList far_near(const shbim_ctx* ctx, const FarPlan& P, int kind);
// target-source pairs of the plan that the kind sums directly (reads the orders back, once per geometry)
double far_direct_pairs(const shbim_ctx* ctx, const FarPlan& P, int kind);
// moments, translations and local expansions from the strengths in dens_up*; then their values at the targets
int far_expand(shbim_ctx* ctx, const FarPlan& P, int kind, cudaStream_t s);
int far_evaluate(shbim_ctx* ctx, const FarPlan& P, int kind, double* out, cudaStream_t s);

}  // namespace shbim
