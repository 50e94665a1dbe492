// varsum.cuh -- finding the slots of one variable (the per-variable kernels of
// kernels_misc.cu and kernels_params.cu): a variable is a thread's, or a warp's
// when it has more than kWide slots.
#pragma once

#include "kernels.h"

namespace dg {

// The first kEll slots of variable i; returns whether there are more.
__device__ __forceinline__ bool ell_slots(const DevArena& A, int i, int (&q)[kEll]) {
#pragma unroll
  for (int r = 0; r < kEll; ++r) q[r] = __ldg(A.var_ell + (int64_t)r * A.n + i);
  const bool more = q[kEll - 1] <= -2;
  if (more) q[kEll - 1] = -2 - q[kEll - 1];
  return more;
}

// Threads per block of the per-variable kernels, blocks over all variables and
// over the wide ones (a warp each).
constexpr int kVarThreads = 256;
inline int var_blocks(const DevArena& A) { return (A.n + kVarThreads - 1) / kVarThreads; }
inline int wide_blocks(const DevArena& A) { return (A.num_wide + kVarThreads / 32 - 1) / (kVarThreads / 32); }

// The variable of a thread (blocks below nblk) or a warp (the others): its
// number, the slots of the ELL columns (threads) and the rest of its list
// [b, e) (a warp's whole list).  `mine`: there is one (else nothing to do).
struct VarWalk {
  int i, b, e, q[kEll], lane;
  bool wide, mine;
};
__device__ __forceinline__ VarWalk var_walk(const DevArena& A, int nblk) {
  VarWalk v;
  v.wide = (int)blockIdx.x >= nblk;
  v.lane = threadIdx.x & 31;
  const int x = (v.wide ? (int)blockIdx.x - nblk : (int)blockIdx.x) * (int)blockDim.x + (int)threadIdx.x;
  v.b = v.e = 0;
#pragma unroll
  for (int r = 0; r < kEll; ++r) v.q[r] = -1;
  if (v.wide) {
    const int w = x >> 5;
    v.mine = w < A.num_wide;  // uniform in the warp
    v.i = v.mine ? __ldg(A.wide_vars + w) : 0;
    v.b = v.mine ? __ldg(A.var_ptr + v.i) : 0;
    v.e = v.mine ? __ldg(A.var_ptr + v.i + 1) : 0;
  } else {
    v.i = x;
    v.mine = x < A.n;
    if (v.mine && ell_slots(A, x, v.q)) {
      v.b = __ldg(A.var_ptr + x) + kEll;
      v.e = __ldg(A.var_ptr + x + 1);
      v.mine = v.e - v.b <= kWide - kEll;  // else a wide variable
    }
  }
  return v;
}
__device__ __forceinline__ int var_degree(const VarWalk& v) {
  int d = v.e - v.b;
#pragma unroll
  for (int r = 0; r < kEll; ++r) d += v.q[r] >= 0;
  return d;
}

}  // namespace dg
