// kernels_misc.cu -- per-variable and per-instance kernels around the sweeps:
// the deferred min-marginal sums S_i (Alg. 1, lambda update), the FP64
// re-projection onto the dual constraint of (D), the initial split of c and
// the FP64 lower bound (Def. 2 with the unary term of the deferred
// min-marginals).
#include "varsum.cuh"

namespace dg {

// x[q] summed over the slots of one variable in fixed order: the first kEll
// slots (q, from the ELL columns, -1 past the end), then var_slots[b .. e).
// The loads of a batch are all issued before its first addition; the order of
// the additions is the plain loop's.
__device__ __forceinline__ float sum_slots(const DevArena& A, const float* x, const int (&q)[kEll], int b, int e) {
  float v[kEll], s = 0.f;
#pragma unroll
  for (int r = 0; r < kEll; ++r) v[r] = q[r] >= 0 ? x[q[r]] : 0.f;
#pragma unroll
  for (int r = 0; r < kEll; ++r)
    if (q[r] >= 0) s += v[r];
  constexpr int kB = 8;
  for (int k = b; k < e; k += kB) {
    int p[kB];
    float w[kB];
#pragma unroll
    for (int j = 0; j < kB; ++j) p[j] = k + j < e ? __ldg(A.var_slots + k + j) : -1;
#pragma unroll
    for (int j = 0; j < kB; ++j) w[j] = p[j] >= 0 ? x[p[j]] : 0.f;
#pragma unroll
    for (int j = 0; j < kB; ++j)
      if (p[j] >= 0) s += w[j];
  }
  return s;
}

// ... by a warp, for the wide variables: the lanes load 32 values at a time
// and every lane adds them in slot order (the same sum to the bit).
__device__ __forceinline__ float sum_slots_warp(const DevArena& A, const float* x, int b, int e, int lane) {
  float s = 0.f;
  for (int c = b; c < e; c += 32) {
    const float v = c + lane < e ? x[__ldg(A.var_slots + c + lane)] : 0.f;
    const int cnt = min(32, e - c);
    for (int j = 0; j < cnt; ++j) s += __shfl_sync(0xffffffffu, v, j);
  }
  return s;
}

// S_i = sum_{j in J_i} M_ij over the variable's slots in fixed order.  Blocks
// below nblk take a variable per thread, the others a wide variable (more than
// kWide slots) per warp.  `need`: whether to store S (kNeedS) and, before a
// sweep (kNeedAvg), the averaging term it adds (S_i / |J_i| in mode 0, S_i in
// mode 1, which it multiplies by alpha_ij).  With SCATTER every slot in
// [from, to) of the variable also receives that term; the unit rows' sweeps
// gather it per variable instead, which halves the reduction's random accesses.
template <bool SCATTER>
__global__ void __launch_bounds__(256) k_reduce_S(DevArena A, const float* M, int mode, int need, int from, int to,
                                                   int nblk) {
  const bool wide = (int)blockIdx.x >= nblk;
  const int lane = threadIdx.x & 31;
  const int x = (wide ? (int)blockIdx.x - nblk : (int)blockIdx.x) * (int)blockDim.x + (int)threadIdx.x;
  int i, b = 0, e = 0, q[kEll] = {-1, -1, -1, -1};
  bool mine = true;
  if (wide) {
    const int w = x >> 5;
    mine = w < A.num_wide;  // uniform in the warp
    i = mine ? __ldg(A.wide_vars + w) : 0;
    b = mine ? __ldg(A.var_ptr + i) : 0;
    e = mine ? __ldg(A.var_ptr + i + 1) : 0;
  } else {
    i = x;
    mine = i < A.n;
    if (mine && ell_slots(A, i, q)) {
      b = __ldg(A.var_ptr + i) + kEll;
      e = __ldg(A.var_ptr + i + 1);
      mine = e - b <= kWide - kEll;  // else a wide variable
    }
  }
  grid_wait();
  grid_trigger();
  if (!mine) return;
  const float s = wide ? sum_slots_warp(A, M, b, e, lane) : sum_slots(A, M, q, b, e);
  const float t = mode == 1 ? s : __ldg(A.invdeg + i) * s;
  if (!wide || lane == 0) {
    if (need & kNeedS) A.S[i] = s;
    if (need & kNeedAvg) A.var_avg[i] = t;
  }
  if (SCATTER) {
    if (!wide) {
#pragma unroll
      for (int r = 0; r < kEll; ++r)
        if (q[r] >= from && q[r] < to) A.slot_avg[q[r]] = t;
    }
    for (int k = b + (wide ? lane : 0); k < e; k += wide ? 32 : 1) {
      const int p = __ldg(A.var_slots + k);
      if (p >= from && p < to) A.slot_avg[p] = t;
    }
  }
}

// The reduction with the re-projection of lambda onto sum_j (lambda_ij + M_ij)
// = c_i (the invariant of the proof of Prop. 1): the FP64 residual
// r_i = c_i - sum_j (lambda_ij + M_ij) is spread with the averaging weights.
template <bool SCATTER>
__global__ void __launch_bounds__(256) k_reduce_renorm(DevArena A, const float* __restrict__ M, float* lam,
                                                        const float* __restrict__ alpha, int mode, int need, int from,
                                                        int to) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.n) return;
  const int b = __ldg(A.var_ptr + i), e = __ldg(A.var_ptr + i + 1);
  float s = 0.f;
  double tot = 0.0;
  for (int k = b; k < e; ++k) {
    const int q = __ldg(A.var_slots + k);
    const float mk = M[q];
    s += mk;
    tot += (double)lam[q] + (double)mk;
  }
  const float inv = __ldg(A.invdeg + i);
  const float t = mode == 1 ? s : inv * s;
  A.S[i] = s;
  if (need & kNeedAvg) A.var_avg[i] = t;
  if (e > b) {
    const double r = A.c[i] - tot;
    for (int k = b; k < e; ++k) {
      const int q = __ldg(A.var_slots + k);
      const double w = mode == 1 ? (double)alpha[q] : (double)inv;
      lam[q] = (float)((double)lam[q] + w * r);
      if (SCATTER && q >= from && q < to) A.slot_avg[q] = t;
    }
  }
}

__global__ void k_init(DevArena A, float* lam, float* M) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= A.num_slots) return;
  const int var = __ldg(A.slot_var + q);
  float l = 0.f;
  if (var >= 0) {
    const int deg = __ldg(A.var_ptr + var + 1) - __ldg(A.var_ptr + var);
    l = (float)(A.c[var] / (double)deg);
  }
  lam[q] = l;
  M[q] = 0.f;
}

// One partial sum per chunk: rows contribute E^j, variables min(0, S_i)
// (variables no row covers add min(0, c_i), a constant per instance that
// k_lb_final adds).  FP64 arithmetic is slow on this
// part, so every thread accumulates its float32 terms with Knuth's TwoSum
// (an error-free transformation: the running sum and its exact rounding
// error, both float32), and only the per-thread results are combined in
// FP64, in a fixed order (deterministic for a given layout).
__global__ void __launch_bounds__(256) k_lb_partial(DevArena A) {
  grid_wait();
  grid_trigger();
  const int4 ch = __ldg(A.lb_chunks + blockIdx.x);
  float hi = 0.f, lo = 0.f;
  // variables no row covers have S_i = 0 (an empty sum), so min(0, S_i) adds
  // nothing for them; their cost term is the per-instance constant inst_unc
  const bool rows = ch.y == 0;
  const float* src = rows ? A.E : A.S;
  constexpr int kU = 4;  // loads of kU elements are issued before their sums
  for (int x0 = ch.z + threadIdx.x; x0 < ch.w; x0 += kU * blockDim.x) {
    float v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int x = x0 + u * blockDim.x;
      const float y = x < ch.w ? src[x] : 0.f;
      v[u] = rows ? y : fminf(0.f, y);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const float s = hi + v[u];
      const float bp = s - hi;
      lo += (hi - (s - bp)) + (v[u] - bp);
      hi = s;
    }
  }
  // float-float tree over the block (TwoSum at every step), one conversion
  // to float64 per block: FP64 arithmetic is slow on this part
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h2 = __shfl_down_sync(0xFFFFFFFFu, hi, o);
    const float l2 = __shfl_down_sync(0xFFFFFFFFu, lo, o);
    const float s = hi + h2;
    const float bp = s - hi;
    lo = lo + l2 + ((hi - (s - bp)) + (h2 - bp));
    hi = s;
  }
  __shared__ float rh[8], rl[8];
  if ((threadIdx.x & 31) == 0) {
    rh[threadIdx.x >> 5] = hi;
    rl[threadIdx.x >> 5] = lo;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += (double)rh[w] + (double)rl[w];
    A.lb_part[blockIdx.x] = t;
  }
}

// One CTA per instance sums the instance's chunk partials (strided per
// thread, then a fixed tree): deterministic for a given layout.
__global__ void __launch_bounds__(256) k_lb_final(DevArena A, double* lb) {
  grid_wait();
  grid_trigger();
  const int k = blockIdx.x;
  double t = 0.0;
  for (int c = A.inst_chunk_ptr[k] + threadIdx.x; c < A.inst_chunk_ptr[k + 1]; c += blockDim.x) t += A.lb_part[c];
  __shared__ double red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xFFFFFFFFu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    lb[k] = s + A.inst_unc[k];
  }
}

__global__ void k_seed_M(DevArena A, float* gM) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= A.num_slots) return;
  const int var = __ldg(A.slot_var + q);
  gM[q] = (var >= 0 && A.S[var] < 0.f) ? 1.f : 0.f;
}

// Between two adjoint sweeps: the S-dot of a variable (sum of its slots'
// contributions) and the inputs of the next adjoint sweep.  Blocks as in
// k_reduce_S.
__global__ void __launch_bounds__(256) k_slot_inputs(DevArena A, const float* x, const float* sd_in, float* out_var,
                                                      const float* S_var, float2* var_in, float2* slot_in, int nblk) {
  const bool wide = (int)blockIdx.x >= nblk;
  const int lane = threadIdx.x & 31;
  const int t = (wide ? (int)blockIdx.x - nblk : (int)blockIdx.x) * (int)blockDim.x + (int)threadIdx.x;
  int i, b = 0, e = 0, q[kEll] = {-1, -1, -1, -1};
  bool mine = true;
  if (wide) {
    const int w = t >> 5;
    mine = w < A.num_wide;
    i = mine ? __ldg(A.wide_vars + w) : 0;
    b = mine ? __ldg(A.var_ptr + i) : 0;
    e = mine ? __ldg(A.var_ptr + i + 1) : 0;
  } else {
    i = t;
    mine = i < A.n;
    if (mine && ell_slots(A, i, q)) {
      b = __ldg(A.var_ptr + i) + kEll;
      e = __ldg(A.var_ptr + i + 1);
      mine = e - b <= kWide - kEll;
    }
  }
  grid_wait();
  grid_trigger();
  if (!mine) return;
  float s = 0.f;
  if (x)
    s = wide ? sum_slots_warp(A, x, b, e, lane) : sum_slots(A, x, q, b, e);
  else if (sd_in)
    s = sd_in[i];
  if (out_var && (!wide || lane == 0)) out_var[i] = s;
  if (var_in) {
    const float2 v = make_float2(s, S_var ? S_var[i] : 0.f);
    if (!wide || lane == 0) var_in[i] = v;
    if (slot_in) {
      if (!wide) {
#pragma unroll
        for (int r = 0; r < kEll; ++r)
          if (q[r] >= A.unit_slots) slot_in[q[r]] = v;
      }
      for (int k = b + (wide ? lane : 0); k < e; k += wide ? 32 : 1) {
        const int p = __ldg(A.var_slots + k);
        if (p >= A.unit_slots) slot_in[p] = v;
      }
    }
  }
}

__global__ void k_slot_invdeg(DevArena A) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= A.num_slots) return;
  const int var = __ldg(A.slot_var + q);
  A.slot_invdeg[q] = var >= 0 ? __ldg(A.invdeg + var) : 0.f;
}

void launch_fill_slot_invdeg(const DevArena& A, cudaStream_t st) {
  const int T = 256;
  const int64_t G = (A.num_slots + T - 1) / T;
  if (G > 0) k_slot_invdeg<<<(unsigned)G, T, 0, st>>>(A);
}

__global__ void k_gather_var(DevArena A, const float* __restrict__ v, float* out) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= A.num_slots) return;
  const int var = __ldg(A.slot_var + q);
  out[q] = var >= 0 ? v[var] : 0.f;
}

// The slots whose averaging term the sweeps read per slot: the mixed tiles',
// and the long BDDs' unless all of them sweep as unit rows.
static int scatter_to(const DevArena& A) {
  return A.num_long == A.long_plain ? A.long_slot_base : (int)A.num_slots;
}

void launch_slot_inputs(const DevArena& A, const float* x, const float* sd_in, float* out_var, const float* S_var,
                        float2* var_in, float2* slot_in, Chain& ch) {
  if (A.unit_slots >= scatter_to(A)) slot_in = nullptr;  // no slot reads it
  const int G = var_blocks(A);
  if (G > 0)
    chain_launch(ch, k_slot_inputs, G + wide_blocks(A), kVarThreads, 0, A, x, sd_in, out_var, S_var, var_in, slot_in, G);
}

void launch_gather_var(const DevArena& A, const float* v, float* out_slot, cudaStream_t st) {
  const int T = 256;
  const int64_t G = (A.num_slots + T - 1) / T;
  if (G > 0) k_gather_var<<<(unsigned)G, T, 0, st>>>(A, v, out_slot);
}

void launch_reduce_S(const DevArena& A, const float* M, float* lam, const float* alpha, int mode, bool renorm,
                     Chain& ch, Scatter to, bool store_S) {
  const int G = var_blocks(A);
  if (G == 0) return;
  const int from = A.unit_slots, end = scatter_to(A);
  const bool scatter = to == Scatter::kSweep && from < end;
  const int need = (store_S ? kNeedS : 0) | (to == Scatter::kSweep ? kNeedAvg : 0);
  if (renorm) {
    ch.linked = false;
    scatter ? k_reduce_renorm<true><<<G, kVarThreads, 0, ch.ss.main>>>(A, M, lam, alpha, mode, need, from, end)
            : k_reduce_renorm<false><<<G, kVarThreads, 0, ch.ss.main>>>(A, M, lam, alpha, mode, need, from, end);
  } else {
    chain_launch(ch, scatter ? k_reduce_S<true> : k_reduce_S<false>, G + wide_blocks(A), kVarThreads, 0, A, M, mode,
                 need, from, end, G);
  }
}

void launch_init(const DevArena& A, float* lam, float* M, cudaStream_t st) {
  const int T = 256;
  const int64_t G = (A.num_slots + T - 1) / T;
  if (G > 0) k_init<<<(unsigned)G, T, 0, st>>>(A, lam, M);
}

void launch_lower_bound(const DevArena& A, double* lb, Chain& ch) {
  if (A.num_lb_chunks > 0) chain_launch(ch, k_lb_partial, A.num_lb_chunks, 256, 0, A);
  chain_launch(ch, k_lb_final, A.num_inst, 256, 0, A, lb);
}

void launch_seed_M(const DevArena& A, float* gM, cudaStream_t st) {
  const int T = 256;
  const int64_t G = (A.num_slots + T - 1) / T;
  if (G > 0) k_seed_M<<<(unsigned)G, T, 0, st>>>(A, gM);
}

}  // namespace dg
