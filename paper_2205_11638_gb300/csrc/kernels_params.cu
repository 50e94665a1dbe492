// kernels_params.cu -- per-variable segmented operations around the solver
// that DOGE-Train's pipeline applies between rounds of Alg. 1:
//  * the non-parametric update of eq. 2 (Sec. 3.4),
//    lambda_ij += theta_ij - mean_{k in J_i} theta_ik, and its adjoint;
//  * the output transforms of the parameter predictor (Alg. 3): softmax of
//    alpha-hat over J_i, sigmoid of omega-hat, centring of theta-hat, and
//    their adjoints.
// A variable is a thread's (its first slots from the coalesced ELL columns, the
// values of all of them in flight together and kept in registers) or, with more
// than kWide slots, a warp's; sums in the fixed order of the variable CSR
// (deterministic).  What needs no variable (sigmoid and its adjoint) runs over
// the slots in blocks of its own, coalesced.  Bound by the uncoalesced accesses
// to the slots; padding slots are never touched.  One thread per variable
// walking its list once per pass against this (us, GB300, tracking with 200
// frames of 2,000 detections / quadratic matching of 200): transforms 139 -> 110
// / 81 -> 30, their adjoint 167 -> 119 / 61 -> 28, the update 176 -> 123 / 43 ->
// 20, centring 50 -> 40 / 21 -> 17; matching was bound by its longest lists.
#include "varsum.cuh"

namespace dg {

namespace {

// The values of x at a variable's first slots, all loads issued at once.
struct Head {
  float v[kEll];
};
__device__ __forceinline__ Head head(const float* x, const VarWalk& w) {
  Head h;
#pragma unroll
  for (int r = 0; r < kEll; ++r) h.v[r] = w.q[r] >= 0 ? x[w.q[r]] : 0.f;
  return h;
}
// f(slot, value of x) over the slots, the first ones' values from h.
template <class F>
__device__ __forceinline__ void each_value(const DevArena& A, const VarWalk& w, const Head& h, const float* x, F&& f) {
#pragma unroll
  for (int r = 0; r < kEll; ++r)
    if (w.q[r] >= 0) f(w.q[r], h.v[r]);
  const int step = w.wide ? 32 : 1;
#pragma unroll 4
  for (int k = w.b + (w.wide ? w.lane : 0); k < w.e; k += step) {
    const int q = __ldg(A.var_slots + k);
    f(q, x[q]);
  }
}
// Sum of f(slot, value) in slot order.
template <class F>
__device__ __forceinline__ float ordered_sum(const DevArena& A, const VarWalk& w, const Head& h, const float* x, F&& f) {
  float s = 0.f;
  if (!w.wide) {
    each_value(A, w, h, x, [&](int q, float v) { s = f(s, q, v); });
    return s;
  }
  for (int c = w.b; c < w.e; c += 32) {
    const int q = c + w.lane < w.e ? __ldg(A.var_slots + c + w.lane) : -1;
    const float v = q >= 0 ? x[q] : 0.f;
    const int cnt = min(32, w.e - c);
    for (int j = 0; j < cnt; ++j) s = f(s, __shfl_sync(0xffffffffu, q, j), __shfl_sync(0xffffffffu, v, j));
  }
  return s;
}
__device__ __forceinline__ float plain_sum(const DevArena& A, const VarWalk& w, const Head& h, const float* x) {
  return ordered_sum(A, w, h, x, [](float s, int, float v) { return s + v; });
}

// out = x - mean over J_i
__device__ __forceinline__ void centre(const DevArena& A, const VarWalk& w, const float* x, float* out) {
  const Head h = head(x, w);
  const float mean = plain_sum(A, w, h, x) / (float)var_degree(w);
  each_value(A, w, h, x, [&](int q, float v) { out[q] = v - mean; });
}

// Blocks past the per-variable ones take the slots, kVarThreads each.
__device__ __forceinline__ int64_t slot_of_block(int first) {
  return (int64_t)((int)blockIdx.x - first) * kVarThreads + threadIdx.x;
}

}  // namespace

__global__ void __launch_bounds__(kVarThreads) k_nonparam(DevArena A, float* lam, const float* __restrict__ theta,
                                                          int nblk) {
  const VarWalk w = var_walk(A, nblk);
  if (!w.mine || var_degree(w) == 0) return;
  const Head h = head(theta, w), l = head(lam, w);
  const float mean = plain_sum(A, w, h, theta) / (float)var_degree(w);
#pragma unroll
  for (int r = 0; r < kEll; ++r)
    if (w.q[r] >= 0) lam[w.q[r]] = l.v[r] + (h.v[r] - mean);
  // the others four at a time: lam may not be read ahead of a store to it
  const int step = w.wide ? 32 : 1;
  for (int k = w.b + (w.wide ? w.lane : 0); k < w.e; k += 4 * step) {
    int q[4];
    float x[4], y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = k + j * step < w.e ? __ldg(A.var_slots + k + j * step) : -1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = q[j] >= 0 ? lam[q[j]] : 0.f;
      y[j] = q[j] >= 0 ? theta[q[j]] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (q[j] >= 0) lam[q[j]] = x[j] + (y[j] - mean);
  }
}

// out = x - mean over J_i (the centring; its own adjoint)
__global__ void __launch_bounds__(kVarThreads) k_center(DevArena A, const float* __restrict__ x, float* out, int nblk) {
  const VarWalk w = var_walk(A, nblk);
  if (!w.mine || var_degree(w) == 0) return;
  centre(A, w, x, out);
}

__global__ void __launch_bounds__(kVarThreads) k_param_transform(DevArena A, const float* __restrict__ ah,
                                                                 const float* __restrict__ wh,
                                                                 const float* __restrict__ th, float* alpha,
                                                                 float* omega, float* theta, int nblk, int vblk) {
  if ((int)blockIdx.x >= vblk) {
    const int64_t q = slot_of_block(vblk);
    if (q < A.num_slots && __ldg(A.slot_var + q) >= 0) omega[q] = 1.0f / (1.0f + expf(-wh[q]));
    return;
  }
  const VarWalk w = var_walk(A, nblk);
  if (!w.mine || var_degree(w) == 0) return;
  if (alpha) {
    Head h = head(ah, w);
    float mx = -3.0e38f;
    each_value(A, w, h, ah, [&](int, float v) { mx = fmaxf(mx, v); });
    if (w.wide)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
    for (int r = 0; r < kEll; ++r) h.v[r] = expf(h.v[r] - mx);  // the first slots' exponentials, once
    float z = 0.f;
    if (!w.wide) {
#pragma unroll
      for (int r = 0; r < kEll; ++r)
        if (w.q[r] >= 0) z += h.v[r];
#pragma unroll 4
      for (int k = w.b; k < w.e; ++k) z += expf(ah[__ldg(A.var_slots + k)] - mx);
    } else {
      for (int c = w.b; c < w.e; c += 32) {
        const float v = c + w.lane < w.e ? expf(ah[__ldg(A.var_slots + c + w.lane)] - mx) : 0.f;
        const int cnt = min(32, w.e - c);
        for (int j = 0; j < cnt; ++j) z += __shfl_sync(0xffffffffu, v, j);
      }
    }
#pragma unroll
    for (int r = 0; r < kEll; ++r)
      if (w.q[r] >= 0) alpha[w.q[r]] = h.v[r] / z;
    const int step = w.wide ? 32 : 1;
#pragma unroll 4
    for (int k = w.b + (w.wide ? w.lane : 0); k < w.e; k += step) {
      const int q = __ldg(A.var_slots + k);
      alpha[q] = expf(ah[q] - mx) / z;
    }
  }
  if (theta) centre(A, w, th, theta);
}

__global__ void __launch_bounds__(kVarThreads) k_param_transform_bwd(DevArena A, const float* __restrict__ alpha,
                                                                     const float* __restrict__ omega,
                                                                     const float* __restrict__ ga,
                                                                     const float* __restrict__ gw,
                                                                     const float* __restrict__ gt, float* gah,
                                                                     float* gwh, float* gth, int nblk, int vblk) {
  if ((int)blockIdx.x >= vblk) {
    const int64_t q = slot_of_block(vblk);
    if (q < A.num_slots && __ldg(A.slot_var + q) >= 0) {
      const float o = omega[q];
      gwh[q] = gw[q] * o * (1.0f - o);
    }
    return;
  }
  const VarWalk w = var_walk(A, nblk);
  if (!w.mine || var_degree(w) == 0) return;
  if (gah) {
    const Head h = head(alpha, w), g = head(ga, w);
    float dot = 0.f;
    if (!w.wide) {
#pragma unroll
      for (int r = 0; r < kEll; ++r)
        if (w.q[r] >= 0) dot += h.v[r] * g.v[r];
#pragma unroll 4
      for (int k = w.b; k < w.e; ++k) {
        const int q = __ldg(A.var_slots + k);
        dot += alpha[q] * ga[q];
      }
    } else {
      for (int c = w.b; c < w.e; c += 32) {
        const int q = c + w.lane < w.e ? __ldg(A.var_slots + c + w.lane) : -1;
        const float x = q >= 0 ? alpha[q] : 0.f, y = q >= 0 ? ga[q] : 0.f;
        const int cnt = min(32, w.e - c);
        for (int j = 0; j < cnt; ++j) dot += __shfl_sync(0xffffffffu, x, j) * __shfl_sync(0xffffffffu, y, j);
      }
    }
#pragma unroll
    for (int r = 0; r < kEll; ++r)
      if (w.q[r] >= 0) gah[w.q[r]] = h.v[r] * (g.v[r] - dot);
    const int step = w.wide ? 32 : 1;
#pragma unroll 4
    for (int k = w.b + (w.wide ? w.lane : 0); k < w.e; k += step) {
      const int q = __ldg(A.var_slots + k);
      gah[q] = alpha[q] * (ga[q] - dot);
    }
  }
  if (gth) centre(A, w, gt, gth);
}

static unsigned slot_blocks(const DevArena& A) { return (unsigned)((A.num_slots + kVarThreads - 1) / kVarThreads); }

void launch_nonparam(const DevArena& A, float* lam, const float* theta, cudaStream_t st) {
  if (A.n > 0) k_nonparam<<<var_blocks(A) + wide_blocks(A), kVarThreads, 0, st>>>(A, lam, theta, var_blocks(A));
}
void launch_center(const DevArena& A, const float* x, float* out, cudaStream_t st) {
  if (A.n > 0) k_center<<<var_blocks(A) + wide_blocks(A), kVarThreads, 0, st>>>(A, x, out, var_blocks(A));
}
void launch_param_transform(const DevArena& A, const float* ah, const float* wh, const float* th, float* alpha,
                            float* omega, float* theta, cudaStream_t st) {
  // one launch, unless an output takes the place of another's input: then one by one
  if ((alpha && (alpha == wh || alpha == th)) || (omega && (omega == ah || omega == th)) ||
      (theta && (theta == ah || theta == wh))) {
    if (alpha) launch_param_transform(A, ah, nullptr, nullptr, alpha, nullptr, nullptr, st);
    if (omega) launch_param_transform(A, nullptr, wh, nullptr, nullptr, omega, nullptr, st);
    if (theta) launch_param_transform(A, nullptr, nullptr, th, nullptr, nullptr, theta, st);
    return;
  }
  const int v = alpha || theta ? var_blocks(A) + wide_blocks(A) : 0;
  const unsigned g = (unsigned)v + (omega ? slot_blocks(A) : 0u);
  if (g > 0) k_param_transform<<<g, kVarThreads, 0, st>>>(A, ah, wh, th, alpha, omega, theta, var_blocks(A), v);
}
void launch_param_transform_bwd(const DevArena& A, const float* alpha, const float* omega, const float* ga,
                                const float* gw, const float* gt, float* gah, float* gwh, float* gth, cudaStream_t st) {
  if ((gah && (gah == omega || gah == gw || gah == gt)) || (gwh && (gwh == alpha || gwh == ga || gwh == gt)) ||
      (gth && (gth == alpha || gth == omega || gth == ga || gth == gw))) {  // as above
    if (gah) launch_param_transform_bwd(A, alpha, nullptr, ga, nullptr, nullptr, gah, nullptr, nullptr, st);
    if (gwh) launch_param_transform_bwd(A, nullptr, omega, nullptr, gw, nullptr, nullptr, gwh, nullptr, st);
    if (gth) launch_param_transform_bwd(A, nullptr, nullptr, nullptr, nullptr, gt, nullptr, nullptr, gth, st);
    return;
  }
  const int v = gah || gth ? var_blocks(A) + wide_blocks(A) : 0;
  const unsigned g = (unsigned)v + (gwh ? slot_blocks(A) : 0u);
  if (g > 0)
    k_param_transform_bwd<<<g, kVarThreads, 0, st>>>(A, alpha, omega, ga, gw, gt, gah, gwh, gth, var_blocks(A), v);
}

}  // namespace dg
