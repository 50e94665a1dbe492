// kernels.h -- host-side launchers of the libdg kernels (internal).
#pragma once

#include <cuda_runtime.h>

#include "dg_internal.h"

namespace dg {

// kFwdRec / kBwdRec: the update sweeps that also record, for the adjoint,
// the argmins of their min-sum recursions (see SweepArgs::rec_*).
enum SweepKind : int { kFwd = 0, kBwd = 1, kMinMarg = 2, kEnergy = 3, kSeed = 4, kFwdRec = 5, kBwdRec = 6 };

struct SweepArgs {
  float* lam;          // in/out (read-only for kMinMarg/kEnergy/kSeed)
  float* M;            // out: M (kFwd/kBwd), m0 (kMinMarg), g_lam (kSeed)
  float* out2;         // out: m1 (kMinMarg)
  const float* omega;  // mode 1
  const float* alpha;  // mode 1
  float omega0;        // mode 0
  int mode;
  float* E;            // nullable: E^j per original row (kBwd, kEnergy)
  // Hand-off of App. B's path costs from one update sweep (plain or
  // recording) to the next (per node and lane of the tiles, in the layout of
  // the child codes; both nullable).  cost_out: the costs of the sweep's own
  // direction under the outgoing lambda, which it computes anyway (SP(r, .)
  // after a forward sweep, SP(., T) after a backward one).  cost_in: the
  // costs opposite to the sweep direction under the incoming lambda (SP(., T)
  // for a forward sweep, SP(r, .) for a backward one), read instead of
  // recomputed; valid when lambda has not changed since the sweep that wrote
  // them.  The two may be the same array: each warp stages its tile's part
  // before it writes it.
  float* cost_out;
  const float* cost_in;
  // kFwdRec / kBwdRec with cost_in: the node records (rec_meta, and
  // rec_lmeta for the long BDDs) of the recording sweep that wrote the costs
  const uint16_t* meta_in;
  const int32_t* lmeta_in;
  // argmin records (kFwdRec, kBwdRec), read back by the adjoint of the sweep:
  uint16_t* rec_meta;  // per node (layout of the child codes): in-arc parent | beta << 8 | hi-choice << 9
  uint16_t* rec_amin;  // per slot: argmin node of m0 | argmin node of m1 << 8
  float* rec_diff;     // per slot: m1 - m0
  // (rec_meta and rec_amin hold the mixed tiles only, from node unit_nodes and
  // slot unit_slots on; a unit tile's records are one word per slot)
  uint32_t* rec_unit;
  // ... for the long BDDs: per node (cost scratch index) in-arc << 1 |
  // hi-choice, per long slot (from long_slot_base) the argmin nodes of m0, m1
  int32_t* rec_lmeta;
  int2* rec_lamin;
  // ... and for the long unit BDDs per long slot (from long_slot_base)
  // long_rec_words words: the unit tiles' word where a lane holds a level, else
  // the out-arc bits of the level, the in-arc bits of the next, and the argmin
  // states
  uint32_t* rec_lunit;
};

// The caller's stream plus kStreams - 1 auxiliary streams of an arena: the
// launch groups of one sweep fork from the caller's stream, run on their
// assigned streams concurrently, and join back before the next step.
struct StreamSet {
  cudaStream_t main = nullptr;
  cudaStream_t aux[kStreams - 1] = {};
  cudaEvent_t fork = nullptr;
  cudaEvent_t join[kStreams - 1] = {};
  bool ready = false;
  int n = kStreams;  // streams in use (1: everything on main)
  cudaStream_t of(int k) const {
    const int j = n > 0 ? k % n : 0;
    return j == 0 || !ready ? main : aux[j - 1];
  }
  void begin() const;  // fork
  void end() const;    // join
};

// One API call's work on a stream.  Kernels that begin with grid_wait() (below)
// are launched through chain_launch: each may start while the one before it
// drains, set up whatever does not depend on it (tile and shape records,
// variable ids, slot lists) and only then wait for it, which hides the launch
// latency that small instances consist of.  `linked`: the stream's last
// operation is such a kernel of this call; anything else enqueued in between
// (a copy, a fork) resets it.  Every chained kernel waits before it ends, so
// that the end of one implies the end of all before it.
struct Chain {
  StreamSet ss;
  bool linked = false;
};
template <class... P, class... X>
void chain_launch(Chain& c, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, X... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c.ss.main;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = c.linked ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
  c.linked = true;
}
#ifdef __CUDACC__
// Waits until the kernels before this one in its chain have ended and their
// results are visible (at once when it was not launched into a chain).  Data
// they wrote is read after it, by loads that are not read-only-cached.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the chain start once every block has come here.
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Kinds of long BDDs an arena has (unit rows, others).
inline int long_launches(const DevArena& A) { return (A.num_long_items > 0) + (A.num_long > A.num_long_unit); }

cudaError_t set_sweep_smem_limit(size_t bytes);
cudaError_t set_unit_smem_limit(size_t bytes);
// The launch of one group of unit tiles (kernels_unit.cu), wpc warps of
// `region` bytes to a CTA.
struct AdjArgs;
void launch_unit(int kind, const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region,
                 Chain& ch);
// `iters` iterations of Alg. 1 on a small arena of unit tiles in one launch
// (energies of the last backward sweep into a.E when not NULL); false, and
// nothing launched, when the arena is not of that kind.
//
// The line: kSmallWork, the groups' estimated work (levels times a level's
// cost, 14 W + 40) plus 1.2 per variable.  One block's iteration costs about
// 2 us plus 0.6 us per 1,000 of it, the chain of launches 7 us whatever the
// variables (us per iteration, one block / chain: set cover 24 x 16, work 2,000
// 3.6 / 8.3; independent set of 400 nodes, 7,300 5.9 / 7.4; tracking 3 x 40 per
// slot, about 20,000 12.3 / 11.2; 20 rows over 2,000 variables 3.1 / 7.1, over
// 8,000 7.4 / 7.2, over 32,000 31.5 / 7.2).
constexpr int64_t kSmallWork = 10000;
bool small_arena(const DevArena& A, const LaunchGroup* groups, int num_groups, size_t smem_cap);
bool launch_small_iterate(const DevArena& A, const SweepArgs& a, const LaunchGroup* groups, int num_groups, int iters,
                          size_t smem_cap, Chain& ch);
void launch_unit_smoothed(const DevArena& A, const float* lam, float a_s, float* E_a, float* marg, const LaunchGroup& G,
                          int wpc, size_t region, cudaStream_t st);
void launch_unit_adjoint(bool forward, const DevArena& A, const AdjArgs& a, const AdjGroup& G, int wpc, size_t region,
                         Chain& ch);
// Dynamic shared memory one CTA may use; launchers put fewer warps in a CTA
// when their tiles need more.
void set_cta_smem_cap(size_t bytes);
int best_warps_per_cta(size_t region, int max_wpc, size_t cta_cap);
void launch_sweep(int kind, const DevArena& A, const SweepArgs& a, int threads, const LaunchGroup* groups,
                  int num_groups, Chain& ch);

// S_i = sum_{k in J_i} M_ik in fixed slot order; with renorm, also
// lambda_ij += alpha_ij * (c_i - sum_k (lambda_ik + M_ik)) computed in FP64.
// Before a sweep (kSweep) also the mode's averaging term, into A.var_avg and,
// for the mixed tiles and the long BDDs that are no unit rows, A.slot_avg: the
// snapshot sweeps read, which a reduction for a bound or a seed (kNone) leaves
// alone.  store_S: whether S itself is read afterwards (always stored by a
// re-projection).
enum class Scatter { kNone, kSweep };
constexpr int kNeedS = 1, kNeedAvg = 2;
void launch_reduce_S(const DevArena& A, const float* M, float* lam, const float* alpha, int mode, bool renorm,
                     Chain& ch, Scatter to, bool store_S = true);
void launch_init(const DevArena& A, float* lam, float* M, cudaStream_t st);
// per-instance FP64 lower bound from A.E and A.S
void launch_lower_bound(const DevArena& A, double* lb_out, Chain& ch);
void launch_seed_M(const DevArena& A, float* g_M, cudaStream_t st);

// Backpropagation through one sweep (kernels_adjoint.cu).
struct AdjArgs {
  const uint16_t* rec_meta;  // the records of the sweep (SweepArgs::rec_*)
  const uint16_t* rec_amin;
  const float* rec_diff;
  const uint32_t* rec_unit;
  const float* S_in;       // S at the start of the sweep (per variable)
  const float* omega;      // mode 1
  const float* alpha;      // mode 1
  float omega0;            // mode 0
  int mode;
  const float* seed_M;     // nullable: gradient of the sweep's M output (per slot)
  const float* sdot_next;  // nullable: S-dot of the next sweep (per variable)
  // per slot: {S-dot of the next sweep, S at the sweep's start} of the
  // slot's variable (launch_slot_inputs), what the tiles' reverse reads
  // instead of gathering per variable (with DevArena::slot_invdeg for the
  // weights of mode 0); the long BDDs use the per-variable arrays above
  const float2* slot_in;
  // the same per variable: the unit tiles gather it
  const float2* var_in;
  float* g_lam;            // in: gradient of lambda after the sweep; out: before
  float* g_omega;          // accumulated (nullable: not computed)
  float* g_alpha;          // accumulated (nullable: not computed)
  float* sdot;             // out: alpha * (gradient of lambda after the sweep), per slot
  // long BDDs: the records of the sweep and per-node gradient scratch of
  // SP(., T) and SP(r, .)
  const int32_t* rec_lmeta;
  const int2* rec_lamin;
  const uint32_t* rec_lunit;
  float* long_a1;
  float* long_a2;
};
cudaError_t set_adjoint_smem_limit(size_t bytes);
void launch_adjoint_sweep(bool forward, const DevArena& A, const AdjArgs& a, const AdjGroup* groups, int num_groups,
                          size_t cta_smem_cap, Chain& ch);
// Per variable i: s_i = sum over the slots q of i of x[q] (fixed order), or
// sd_in[i] when x is NULL (0 when both are); out_var[i] = s_i (nullable);
// and, when var_in is not NULL, {s_i, S_var[i] (0 if NULL)} in var_in[i] and
// in slot_in[q] for every slot q >= unit_slots of i (the unit tiles gather
// var_in, the mixed tiles read slot_in).
void launch_slot_inputs(const DevArena& A, const float* x, const float* sd_in, float* out_var, const float* S_var,
                        float2* var_in, float2* slot_in, Chain& ch);
// A.slot_invdeg[q] = 1/|J_i| of the variable of slot q (0 for padding)
void launch_fill_slot_invdeg(const DevArena& A, cudaStream_t st);
// out_slot[q] = v[variable of q] (0 for padding slots)
void launch_gather_var(const DevArena& A, const float* v, float* out_slot, cudaStream_t st);

// smoothed subproblems (soft-min reading) and their marginals
void launch_smoothed(const DevArena& A, const float* lam, float a_s, float* E_a, float* marg, const LaunchGroup* groups,
                     int num_groups, const StreamSet& ss);

// eq. 2 and the output transforms of Alg. 3 (kernels_params.cu)
void launch_nonparam(const DevArena& A, float* lam, const float* theta, cudaStream_t st);
void launch_center(const DevArena& A, const float* x, float* out, cudaStream_t st);
void launch_param_transform(const DevArena& A, const float* ah, const float* wh, const float* th, float* alpha,
                            float* omega, float* theta, cudaStream_t st);
void launch_param_transform_bwd(const DevArena& A, const float* alpha, const float* omega, const float* ga,
                                const float* gw, const float* gt, float* gah, float* gwh, float* gth, cudaStream_t st);

// Long BDDs, one warp per BDD (kernels_long.cu); each is a single launch on
// the given stream, or nothing when the arena has no long BDDs.
cudaError_t set_long_smem_limit(size_t bytes);
cudaError_t set_long_unit_smem_limit(size_t bytes);
void launch_long_unit(int kind, const DevArena& A, const SweepArgs& a, Chain& ch);
void launch_long_unit_adjoint(bool forward, const DevArena& A, const AdjArgs& a, Chain& ch);
void launch_long_sweep(int kind, const DevArena& A, const SweepArgs& a, cudaStream_t st);
// Kernels of one sweep over the long BDDs (those of the unit rows included).
int long_sweep_kernels(const DevArena& A, bool plain);
void launch_long_smoothed(const DevArena& A, const float* lam, float a_s, float* E_a, float* marg, cudaStream_t st);
void launch_long_adjoint(bool forward, const DevArena& A, const AdjArgs& a, cudaStream_t st);

// dg_lower_bound with its intermediates in a static device array (noalloc.cu).
dg_status lower_bound_noalloc(const DevArena& arena, const LaunchGroup* groups, int num_groups, int threads,
                              Chain& ch, const float* lam, const float* M, double* lb);

}  // namespace dg
