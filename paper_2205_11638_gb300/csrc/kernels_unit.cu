// kernels_unit.cu -- the sweeps of Alg. 1, the min-marginals, energies and
// minimising assignments on the unit tiles: rows with coefficients +1 and -1
// (set cover, independent set, at-most-one, flow conservation, linearised
// products), the bulk of the paper's workloads.  See UnitShape for the
// structure and unit.cuh for the recursions.
//
// A sweep reads lambda, a variable id and (through it) the variable's
// averaging term per slot and writes lambda and M; the path costs opposite to
// the sweep are recomputed by a first pass (two operations per state), which
// is cheaper than moving 8 bytes per state through HBM.
//
// Measured against the node-by-node kernel of the mixed tiles (GB300, CUDA
// events, the S reductions included): tracking 500 x 2,000, 50 iterations
// 33.0 -> 22.2 ms; tracking 50 x 400 with per-slot parameters, 100 iterations
// 10.5 -> 3.4 ms; 64 instances batched, 50 iterations 15.0 -> 11.1 ms.
#include "kernels.h"
#include "unit.cuh"

namespace dg {

namespace {

// One tile.  KIND: kFwd, kBwd, kMinMarg, kEnergy, kSeed.
template <int KIND, int MODE, int W>
__device__ __forceinline__ void unit_tile(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                          unsigned char* smem, int lane) {
  constexpr bool UPDATE = KIND == kFwd || KIND == kBwd;
  const UnitCtx s{S.k, S.start, S.accept, S.nruns, A.unit_runs + S.run_base};
  const int64_t sb = T.slot_base;
  const int k = s.k, ns = k * kWarp;
  const bool real = lane < T.nbdd;
  float* lam = (float*)smem;
  float* avg = lam + ns;
  float* om = avg + ns;
  float* al = om + (MODE == 1 ? ns : 0);
  float* cost = UPDATE ? al + ns : avg;  // level h >= 1 at cost + (h - 1) 32 W
  if (MODE == 0) cost = UPDATE ? avg + ns : avg;
  auto row = [&](int h) { return cost + (h - 1) * (kWarp * W); };

  copy_async(lam, a.lam + sb, ns * 4, lane);
  if (UPDATE && MODE == 1) {
    copy_async(om, a.omega + sb, ns * 4, lane);
    copy_async(al, a.alpha + sb, ns * 4, lane);
  }
  cp_async_commit();
  if (UPDATE) {
    // the averaging term of every slot, gathered per variable: it is not
    // needed before the second pass
    const float* src = MODE == 1 ? A.S : A.Sbar;
    const int32_t* var = A.slot_var + sb + lane;
#pragma unroll 4
    for (int h = 0; h < k; ++h) {
      const int v = __ldg(var + h * kWarp);
      if (v >= 0) cp_async4(avg + h * kWarp + lane, src + v);
    }
    cp_async_commit();
    cp_async_wait_one();
  } else {
    cp_async_wait_all();
  }
  __syncwarp();

  if (KIND == kFwd || KIND == kMinMarg) {
    Costs<W> t = unit_end<W>(s.accept);
    unit_levels_up(s, 1, [&](auto ty, int h) {
      t = unit_up<W, decltype(ty)::value>(t, lam[h * kWarp + lane]);
      unit_store<W>(row(h), t, lane);
    });
    if (UPDATE) {
      cp_async_wait_all();
      __syncwarp();
    }
    Costs<W> R = unit_root<W>(s.start);
    unit_levels_down(s, 0, k, [&](auto ty, int h) {
      constexpr int TY = decltype(ty)::value;
      const Costs<W> t1 = h + 1 < k ? unit_load<W>(row(h + 1), lane) : unit_end<W>(s.accept);
      const int q = h * kWarp + lane;
      const float l = lam[q];
      float b0, b1;
      unit_minima<W, TY>(R, t1, b0, b1);
      const float m0 = b0, m1 = l + b1;
      float ln = l;
      if (KIND == kMinMarg) {
        if (real) {
          a.M[sb + q] = m0;
          a.out2[sb + q] = m1;
        }
      } else {
        const float Mn = __fmul_rn(MODE == 1 ? om[q] : a.omega0, m1 - m0);
        ln = unit_lambda_new<MODE>(l, Mn, MODE == 1 ? al[q] : 0.0f, avg[q]);
        if (real) {
          a.lam[sb + q] = ln;
          a.M[sb + q] = Mn;
        }
      }
      R = unit_down<W, TY>(R, ln);
    });
  } else if (KIND == kBwd) {
    Costs<W> R = unit_root<W>(s.start);
    unit_levels_down(s, 0, k - 1, [&](auto ty, int h) {
      R = unit_down<W, decltype(ty)::value>(R, lam[h * kWarp + lane]);
      unit_store<W>(row(h + 1), R, lane);
    });
    cp_async_wait_all();
    __syncwarp();
    Costs<W> t = unit_end<W>(s.accept);
    unit_levels_up(s, 0, [&](auto ty, int h) {
      constexpr int TY = decltype(ty)::value;
      const Costs<W> r = h > 0 ? unit_load<W>(row(h), lane) : unit_root<W>(s.start);
      const int q = h * kWarp + lane;
      const float l = lam[q];
      float b0, b1;
      unit_minima<W, TY>(r, t, b0, b1);
      const float m0 = b0, m1 = l + b1;
      const float Mn = __fmul_rn(MODE == 1 ? om[q] : a.omega0, m1 - m0);
      const float ln = unit_lambda_new<MODE>(l, Mn, MODE == 1 ? al[q] : 0.0f, avg[q]);
      if (real) {
        a.lam[sb + q] = ln;
        a.M[sb + q] = Mn;
      }
      t = unit_up<W, TY>(t, ln);
    });
    if (a.E != nullptr && real) {
      float e = f_inf();  // SP(r, T) = E^j
#pragma unroll
      for (int u = 0; u < W; ++u)
        if (u == s.start) e = t.v[u];
      a.E[__ldg(A.slot_row + sb + lane)] = e;
    }
  } else {
    Costs<W> t = unit_end<W>(s.accept);
    unit_levels_up(s, 0, [&](auto ty, int h) {
      t = unit_up<W, decltype(ty)::value>(t, lam[h * kWarp + lane]);
      if (KIND == kSeed && h > 0) unit_store<W>(row(h), t, lane);
    });
    if (KIND == kEnergy && a.E != nullptr && real) {
      float e = f_inf();
#pragma unroll
      for (int u = 0; u < W; ++u)
        if (u == s.start) e = t.v[u];
      a.E[__ldg(A.slot_row + sb + lane)] = e;
    }
    if (KIND == kSeed) {
      // walk the minimising path from the root: 0-arc on ties
      int at = s.start;
      unit_levels_down(s, 0, k, [&](auto ty, int h) {
        constexpr int TY = decltype(ty)::value;
        const Costs<W> t1 = h + 1 < k ? unit_load<W>(row(h + 1), lane) : unit_end<W>(s.accept);
        const int q = h * kWarp + lane;
        float c0 = f_inf(), c1 = f_inf();
        int z = 0, o = 0;
#pragma unroll
        for (int u = 0; u < W; ++u)
          if (u == at) {
            c0 = t1.at(unit_z<TY>(u));
            c1 = t1.at(unit_o<TY>(u));
            z = unit_z<TY>(u);
            o = unit_o<TY>(u);
          }
        // an infinite cost is the bottom terminal (the path stays feasible)
        const bool take0 = c0 < f_inf() && (c1 == f_inf() || c0 <= lam[q] + c1);
        if (real) a.M[sb + q] = take0 ? 0.f : 1.f;
        at = take0 ? z : o;
      });
    }
  }
}

template <int KIND, int MODE, int WMAX>
__global__ void __launch_bounds__(128) k_unit(DevArena A, SweepArgs a, int region_bytes, int tile0, int tile1) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + warp;
  if (tile >= tile1) return;  // whole warp leaves; no CTA-wide barrier follows
  const Tile T = A.tiles[tile];
  const UnitShape S = A.unit_shapes[T.unit - 1];
  unsigned char* p = smem + (size_t)warp * region_bytes;
  if (S.W == 2)
    unit_tile<KIND, MODE, 2>(A, a, T, S, p, lane);
  else if (WMAX >= 4 && S.W == 4)
    unit_tile<KIND, MODE, 4>(A, a, T, S, p, lane);
  else if (WMAX >= 8 && S.W == 6)
    unit_tile<KIND, MODE, 6>(A, a, T, S, p, lane);
  else if (WMAX >= 8)
    unit_tile<KIND, MODE, 8>(A, a, T, S, p, lane);
}

template <int KIND, int MODE, int WMAX>
void launch_w(const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region, cudaStream_t st) {
  const int nt = G.tile1 - G.tile0;
  k_unit<KIND, MODE, WMAX><<<(nt + wpc - 1) / wpc, wpc * kWarp, region * wpc, st>>>(A, a, (int)region, G.tile0, G.tile1);
}

template <int KIND, int MODE>
void launch_group(const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region,
                  cudaStream_t st) {
  if (G.unit_w <= 2)
    launch_w<KIND, MODE, 2>(A, a, G, wpc, region, st);
  else if (G.unit_w <= 4)
    launch_w<KIND, MODE, 4>(A, a, G, wpc, region, st);
  else
    launch_w<KIND, MODE, 8>(A, a, G, wpc, region, st);
}

template <int KIND, int MODE>
cudaError_t set_attr(int b) {
  cudaError_t e = cudaFuncSetAttribute(k_unit<KIND, MODE, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit<KIND, MODE, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit<KIND, MODE, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  return e;
}

}  // namespace

cudaError_t set_unit_smem_limit(size_t bytes) {
  const int b = (int)bytes;
  cudaError_t e = set_attr<kFwd, 0>(b);
  if (e == cudaSuccess) e = set_attr<kFwd, 1>(b);
  if (e == cudaSuccess) e = set_attr<kBwd, 0>(b);
  if (e == cudaSuccess) e = set_attr<kBwd, 1>(b);
  if (e == cudaSuccess) e = set_attr<kMinMarg, 0>(b);
  if (e == cudaSuccess) e = set_attr<kEnergy, 0>(b);
  if (e == cudaSuccess) e = set_attr<kSeed, 0>(b);
  return e;
}

void launch_unit(int kind, const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region,
                 cudaStream_t st) {
  const bool m1 = a.mode == 1;
  switch (kind) {
    case kFwd: m1 ? launch_group<kFwd, 1>(A, a, G, wpc, region, st) : launch_group<kFwd, 0>(A, a, G, wpc, region, st); break;
    case kBwd: m1 ? launch_group<kBwd, 1>(A, a, G, wpc, region, st) : launch_group<kBwd, 0>(A, a, G, wpc, region, st); break;
    case kMinMarg: launch_group<kMinMarg, 0>(A, a, G, wpc, region, st); break;
    case kEnergy: launch_group<kEnergy, 0>(A, a, G, wpc, region, st); break;
    default: launch_group<kSeed, 0>(A, a, G, wpc, region, st); break;
  }
}

}  // namespace dg
