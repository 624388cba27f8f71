// Plans and workspaces of the expansions between well-separated drops (far.cu).
#pragma once

#include <cstdint>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"

namespace shbim {

constexpr int kFarLmax = 63;        // orders the constant tables hold
constexpr double kFarEps32 = 1e-8;  // truncation of a pair, FP32 sums
constexpr double kFarEps64 = 3e-15; // ... and FP64-class sums
constexpr int kFarCap32 = 36;       // largest order of a far pair, FP32 sums
constexpr int kFarCap64 = 60;       // ... and FP64-class sums
constexpr int kFarPlans = 6;        // [truncation level 2][derivatives 3]

// charge sets of the moments: Laplace strengths; f, y.f; dipole tensor and vector; both
enum FarMode { kFarLap = 0, kFarS = 1, kFarD = 2, kFarSD = 3 };

inline bool stokes_like(int kind) { return kind >= 2; }

struct FarPair {
  int i, j, L, pad;
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

// Per target drop i the drops that no local expansion covers, entries [off[i], off[i+1]): drop index and the number
// of sources before it in the list; the last entry of a drop has index -1 and the total. The targets of a drop are
// taken in the order tgt[] (patches of the surface); group g of 32 of them reaches the multipole expansion of the
// entry's drop at order order[goff[entry] + g] (kNoReach: at none), and is summed directly where that is not worth it.
struct NearList {
  const int* off = nullptr;
  const int* drop = nullptr;
  const int64_t* pre = nullptr;
  const int* tgt = nullptr;
  const int64_t* goff = nullptr;    // [entries + 1]
  const unsigned char* order = nullptr;   // null: every group directly
  FarReach reach;
  __host__ __device__ bool direct(int entry, int group, int ns) const {
    if (!order) return true;
    const int L = order[goff[entry] + group];
    return L == kNoReach || !reach.worth(L, ns);
  }
};

template <class T>
struct FarTab {
  const T *dq_r, *dq_c, *tr, *kap, *rec, *la, *lp, *lq;
  const int *dq_off, *tr_off;
  const int2 *pat_r, *pat_c;
};

struct FarPlan {
  NearList near;
  double direct_pairs = 0.0, far_pairs = 0.0;
  double src_work = 0.0, tgt_work = 0.0, pair_work = 0.0;
  int npairs = 0, nchunks = 0, nblocks = 0, lmax = 0;
  int64_t part = 0, coef = 0, loc = 0, lout = 0, tri = 0, ang = 0;
  bool use[3][5] = {};                // [precision][kind]
  const FarPair* pairs = nullptr;
  const int* Lsrc = nullptr;
  const FarSrcDrop* sd = nullptr;
  const FarTgtDrop* td = nullptr;
  const FarChunk* chunks = nullptr;
  const int2* blocks = nullptr;
  double* ang_dev = nullptr;
  // close pairs: groups of targets far enough for the source drop's own expansion
  int nent = 0;
  int64_t ngroup = 0, stri = 0;
  const int* ent_tgt = nullptr;       // target drop of an entry (-1: end of a list)
  const float* rho_max = nullptr;     // [cap + 1]
  unsigned char* order = nullptr;     // [ngroup]
  std::vector<int> h_drop, h_tgt;     // host copies of the lists
  std::vector<int64_t> h_goff;
  // pairs summed directly, by [precision][kind], once they have been asked for
  mutable bool counted[3][5] = {};
  mutable double count[3][5] = {};
};

struct FarState {
  FarPlan plan[kFarPlans + 1];        // the last one: every other drop directly
  unsigned char* blob = nullptr;      // device copies of the lists of all plans
  size_t blob_cap = 0;
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
  int max_charges = 0;
};

int build_far(shbim_ctx* ctx, const std::vector<double>& ext, cudaStream_t s);
void far_free(shbim_ctx* ctx);
// empties every plan (the workspaces stay): what comes before build_far may fail
void far_forget(shbim_ctx* ctx);
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
