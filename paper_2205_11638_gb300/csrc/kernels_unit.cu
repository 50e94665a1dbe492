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

// A warp's slice of shared memory: per level and lane lambda, (update sweeps)
// the averaging term, (mode 1) omega and alpha, then the path costs of levels
// 1 .. k-1, 32 W floats each.
struct UnitSmem {
  float *lam, *avg, *om, *al, *cost;
};

template <bool UPDATE, int MODE>
__device__ __forceinline__ UnitSmem carve_unit(unsigned char* p, int ns) {
  UnitSmem m;
  m.lam = (float*)p;
  m.avg = m.lam + ns;
  m.om = m.avg + ns;
  m.al = m.om + ns;
  m.cost = !UPDATE ? m.avg : (MODE == 1 ? m.al + ns : m.om);
  return m;
}

// Starts the copies of a tile's inputs.  The variable ids come first, into the
// words of the averaging terms, so that gather_avg can follow as soon as they
// are there: two memory latencies per tile whatever its length (loading the
// ids into registers instead takes one per few levels).
template <bool UPDATE, int MODE>
__device__ __forceinline__ void stage_unit(const DevArena& A, const SweepArgs& a, const UnitSmem& m, int64_t sb,
                                           int ns, int lane) {
  if (UPDATE) {
    copy_async(m.avg, A.slot_var + sb, ns * 4, lane);
    cp_async_commit();
  }
  copy_async(m.lam, a.lam + sb, ns * 4, lane);
  if (UPDATE && MODE == 1) {
    copy_async(m.om, a.omega + sb, ns * 4, lane);
    copy_async(m.al, a.alpha + sb, ns * 4, lane);
  }
  cp_async_commit();
}

// Replaces the staged variable ids by the averaging terms (S_i in mode 1,
// S_i / |J_i| in mode 0), asynchronously: they are not needed before the
// second pass.
template <int MODE>
__device__ __forceinline__ void gather_avg(const DevArena& A, const UnitSmem& m, int ns, int lane) {
  const float* src = MODE == 1 ? A.S : A.Sbar;
#pragma unroll 4
  for (int q = lane; q < ns; q += kWarp) {
    const int v = __float_as_int(m.avg[q]);
    if (v >= 0) cp_async4(m.avg + q, src + v);
  }
  cp_async_commit();
}

// One tile whose inputs are on their way.  KIND: kFwd, kBwd, kMinMarg,
// kEnergy, kSeed.
template <int KIND, int MODE, int W>
__device__ __forceinline__ void unit_tile(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                          const UnitSmem& m, int lane) {
  constexpr bool UPDATE = KIND == kFwd || KIND == kBwd;
  const UnitCtx s{S.k, S.start, S.accept, S.nruns, A.unit_runs + S.run_base};
  const int64_t sb = T.slot_base;
  const int k = s.k;
  const bool real = lane < T.nbdd;
  const float *lam = m.lam, *avg = m.avg, *om = m.om, *al = m.al;
  auto energy = [&](const Costs<W>& t) {  // SP(r, T) = E^j
    float e = f_inf();
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (u == s.start) e = t.v[u];
    a.E[__ldg(A.slot_row + sb + lane)] = e;
  };
  // the update of level h from its minima; returns lambda^new
  auto update = [&](int h, float l, float b0, float b1) -> float {
    const int q = h * kWarp + lane;
    const float m0 = b0, m1 = l + b1;
    const float Mn = __fmul_rn(MODE == 1 ? om[q] : a.omega0, m1 - m0);
    const float ln = unit_lambda_new<MODE>(l, Mn, MODE == 1 ? al[q] : 0.0f, avg[q]);
    if (real) {
      a.lam[sb + q] = ln;
      a.M[sb + q] = Mn;
    }
    return ln;
  };

  if (KIND == kFwd || KIND == kMinMarg) {
    unit_first_up<W>(s, S.rows, lam, m.cost, lane);
    if (UPDATE) cp_async_wait_all();  // every lane gathered its own averaging terms
    Costs<W> R = unit_root<W>(s.start);
    unit_second_down<W>(s, lam, m.cost, lane, [&](auto ty, int h, const Costs<W>& t1) {
      constexpr int TY = decltype(ty)::value;
      const int q = h * kWarp + lane;
      const float l = lam[q];
      float b0, b1;
      unit_minima<W, TY>(R, t1, b0, b1);
      float ln = l;
      if (KIND == kMinMarg) {
        if (real) {
          a.M[sb + q] = b0;
          a.out2[sb + q] = l + b1;
        }
      } else {
        ln = update(h, l, b0, b1);
      }
      R = unit_down<W, TY>(R, ln);
    });
  } else if (KIND == kBwd) {
    unit_first_down<W>(s, lam, m.cost, lane);
    cp_async_wait_all();
    Costs<W> t = unit_end<W>(s.accept);
    unit_second_up<W>(s, S.rows, lam, m.cost, lane, [&](auto ty, int h, const Costs<W>& r) {
      constexpr int TY = decltype(ty)::value;
      const float l = lam[h * kWarp + lane];
      float b0, b1;
      unit_minima<W, TY>(r, t, b0, b1);
      t = unit_up<W, TY>(t, update(h, l, b0, b1));
    });
    if (a.E != nullptr && real) energy(t);
  } else if (KIND == kEnergy) {
    Costs<W> t = unit_end<W>(s.accept);
    unit_runs_up(s, [&](auto ty, int b, int e) {
      for (int h = e - 1; h >= b; --h) t = unit_up<W, decltype(ty)::value>(t, lam[h * kWarp + lane]);
    });
    if (a.E != nullptr && real) energy(t);
  } else {
    // kSeed: walk the minimising path from the root, the 0-arc on ties
    unit_first_up<W>(s, S.rows, lam, m.cost, lane);
    int at = s.start;
    unit_second_down<W>(s, lam, m.cost, lane, [&](auto ty, int h, const Costs<W>& t1) {
      constexpr int TY = decltype(ty)::value;
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

template <int KIND, int MODE, int WMAX>
__global__ void __launch_bounds__(128) k_unit(DevArena A, SweepArgs a, int region_bytes, int tile0, int tile1) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + warp;
  if (tile >= tile1) return;  // whole warp leaves; no CTA-wide barrier follows
  constexpr bool UPDATE = KIND == kFwd || KIND == kBwd;
  const Tile T = A.tiles[tile];
  const int ns = T.nhops * kWarp;
  const UnitSmem m = carve_unit<UPDATE, MODE>(smem + (size_t)warp * region_bytes, ns);
  stage_unit<UPDATE, MODE>(A, a, m, T.slot_base, ns, lane);
  const UnitShape S = A.unit_shapes[T.unit - 1];
  if (UPDATE) {
    cp_async_wait_one();
    __syncwarp();
    gather_avg<MODE>(A, m, ns, lane);
    cp_async_wait_one();
  } else {
    cp_async_wait_all();
  }
  __syncwarp();
  if (S.W == 2)
    unit_tile<KIND, MODE, 2>(A, a, T, S, m, lane);
  else if (WMAX >= 4 && S.W == 4)
    unit_tile<KIND, MODE, 4>(A, a, T, S, m, lane);
  else if (WMAX >= 8 && S.W == 6)
    unit_tile<KIND, MODE, 6>(A, a, T, S, m, lane);
  else if (WMAX >= 8)
    unit_tile<KIND, MODE, 8>(A, a, T, S, m, lane);
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
