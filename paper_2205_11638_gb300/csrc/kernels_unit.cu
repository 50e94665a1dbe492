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
// Before these kernels, with the node-by-node kernel of the mixed tiles, and
// now (GB300, wall clock, the S reductions included): tracking 500 x 2,000, 50
// iterations 33.0 -> 17.9 ms; tracking 50 x 400 with per-slot parameters, 100
// iterations 10.5 -> 1.6 ms; 64 instances batched, 50 iterations 15.3 -> 8.4 ms.
// No unit is saturated: the launches of six and eight states issue in 21 to 30 %
// of the slots at 17 to 44 % of the warps, DRAM at 11 to 15 % and L1 at 22 to
// 31 % of their rates; the tiles wait for their ids, then for the gather of the
// averaging terms, with as few warps as shared memory leaves.
#include <algorithm>

#include "kernels.h"
#include "unit.cuh"

namespace dg {

namespace {

// A warp's slice of shared memory: per level 32 lambdas and (update sweeps) 32
// averaging terms, (mode 1) 32 omegas and 32 alphas, so that one pointer walks
// them all; then the path costs the sweep keeps, 32 W floats per level.
constexpr int kAvg = kWarp, kOm = 2 * kWarp, kAl = 3 * kWarp;
template <bool UPDATE, int MODE>
constexpr int kStride = kWarp * (!UPDATE ? 1 : (MODE == 1 ? 4 : 2));

// k rows of 128 bytes from src to every STRIDE-th float of dst, asynchronously.
template <int STRIDE>
__device__ __forceinline__ void copy_rows(float* dst, const void* src, int k, int lane, uint64_t pol) {
  const char* g = reinterpret_cast<const char*>(src) + lane * 16;
  char* d = reinterpret_cast<char*>(dst) + (lane >> 3) * (STRIDE * 4) + (lane & 7) * 16;
  for (int h = lane >> 3; h < k; h += 4) {
    cp_async16(d, g, pol);
    d += 4 * STRIDE * 4;
    g += 512;
  }
}

// One tile whose inputs are on their way.  KIND: kFwd, kBwd, their recording
// variants kFwdRec and kBwdRec, kMinMarg, kEnergy, kSeed.
template <int KIND, int MODE, int W>
__device__ __forceinline__ void unit_tile(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                          float* smem, int lane) {
  constexpr bool REC = KIND == kFwdRec || KIND == kBwdRec;
  constexpr bool FWD = KIND == kFwd || KIND == kFwdRec;
  constexpr bool BWD = KIND == kBwd || KIND == kBwdRec;
  constexpr bool UPDATE = FWD || BWD;
  constexpr int STRIDE = kStride<UPDATE, MODE>;
  const UnitCtx s{S.k, S.start, S.accept, S.nruns, A.unit_runs + S.run_base};
  const int64_t sb = T.slot_base + lane;
  const bool real = lane < T.nbdd;
  const float* x0 = smem + lane;
  float* cost = smem + s.k * STRIDE;
  auto energy = [&](const Costs<W>& t) {  // SP(r, T) = E^j
    float e = f_inf();
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (u == s.start) e = t.v[u];
    a.E[__ldg(A.slot_row + sb)] = e;
  };
  // where the sweep leaves the level at hand
  const int64_t first = sb + (BWD ? s.k * kWarp : 0);
  float* g0 = (KIND == kMinMarg ? a.out2 : a.lam) + first;
  float* g1 = a.M + first;
  float* gd = REC ? a.rec_diff + first : nullptr;
  uint32_t* gr = REC ? a.rec_unit + first : nullptr;
  auto move = [&](int by) {
    g0 += by;
    g1 += by;
    if (REC) {
      gd += by;
      gr += by;
    }
  };
  // the update of a level from its minima; returns lambda^new
  auto update = [&](const float* x, float b0, float b1) -> float {
    const float l = x[0];
    const float m0 = b0, m1 = l + b1;
    const float Mn = __fmul_rn(MODE == 1 ? x[kOm] : a.omega0, m1 - m0);
    const float ln = unit_lambda_new<MODE>(l, Mn, MODE == 1 ? x[kAl] : 0.0f, x[kAvg]);
    if (real) {
      *g0 = ln;
      *g1 = Mn;
      if (REC) *gd = m1 - m0;
    }
    return ln;
  };

  if (FWD || KIND == kMinMarg) {
    unit_first_up<W, STRIDE>(s, S.rows, x0, cost, lane);
    if (UPDATE) cp_async_wait_all();  // every lane gathered its own averaging terms
    Costs<W> R = unit_root<W>(s.start);
    unit_second_down<W, STRIDE>(s, x0, cost, lane, [&](auto ty, const float* x, const Costs<W>& t1) {
      constexpr int TY = decltype(ty)::value;
      float b0, b1;
      const float l = x[0];
      if (REC) {
        // the out-arcs under the incoming lambda, the in-arcs under the new one
        uint32_t rec = 0;
        unit_minima_rec<W, TY>(R, t1, b0, b1, rec);
        unit_up_rec<W, TY>(t1, l, rec);
        R = unit_down_rec<W, TY>(R, update(x, b0, b1), rec);
        if (real) *gr = rec;
      } else {
        unit_minima<W, TY>(R, t1, b0, b1);
        float ln = l;
        if (KIND == kMinMarg) {
          if (real) {
            *g0 = l + b1;
            *g1 = b0;
          }
        } else {
          ln = update(x, b0, b1);
        }
        R = unit_down<W, TY>(R, ln);
      }
      move(kWarp);
    });
  } else if (BWD) {
    unit_first_down<W, STRIDE>(s, x0, cost, lane);
    cp_async_wait_all();
    Costs<W> t = unit_end<W>(s.accept);
    unit_second_up<W, STRIDE>(s, S.rows, x0, cost, lane, [&](auto ty, const float* x, const Costs<W>& r) {
      constexpr int TY = decltype(ty)::value;
      float b0, b1;
      move(-kWarp);
      if (REC) {
        // the in-arcs under the incoming lambda, the out-arcs under the new one
        uint32_t rec = 0;
        unit_minima_rec<W, TY>(r, t, b0, b1, rec);
        unit_down_rec<W, TY>(r, x[0], rec);
        t = unit_up_rec<W, TY>(t, update(x, b0, b1), rec);
        if (real) *gr = rec;
      } else {
        unit_minima<W, TY>(r, t, b0, b1);
        t = unit_up<W, TY>(t, update(x, b0, b1));
      }
    });
    if (a.E != nullptr && real) energy(t);
  } else if (KIND == kEnergy) {
    Costs<W> t = unit_end<W>(s.accept);
    const float* x = x0 + s.k * STRIDE;
    unit_runs_up(s, [&](auto ty, int b, int e) {
      for (int n = e - b; n > 0; --n) t = unit_up<W, decltype(ty)::value>(t, *(x -= STRIDE));
    });
    if (a.E != nullptr && real) energy(t);
  } else {
    // kSeed: walk the minimising path from the root, the 0-arc on ties
    unit_first_up<W, STRIDE>(s, S.rows, x0, cost, lane);
    int at = s.start;
    unit_second_down<W, STRIDE>(s, x0, cost, lane, [&](auto ty, const float* x, const Costs<W>& t1) {
      constexpr int TY = decltype(ty)::value;
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
      const bool take0 = c0 < f_inf() && (c1 == f_inf() || c0 <= x[0] + c1);
      if (real) *g1 = take0 ? 0.f : 1.f;
      g1 += kWarp;
      at = take0 ? z : o;
    });
  }
}

// ---- short tiles of two states ---------------------------------------------
// Rows of up to kShortK variables with two states a level (pairs of an
// independent set, linearised products, at-most-one and covering rows of a few
// variables) are most tiles of most instances, and a level of theirs is some
// fifteen operations: the staging, loops and run bookkeeping of k_unit were
// four times that.  Here a tile's levels are unrolled, everything is registers,
// and all loads are issued before the first operation, past L1, which is left
// to the gathers (batch of 64: 175 -> 172 us an iteration).  Bound by the latency
// of the ids, then the gathers.  Batch of 64 mixed instances: 189 -> 168 us an
// iteration.  Rows of four variables as well made tracking slower (500 frames,
// 361 -> 386 us), hence kShortK = 3.
template <int TYPE>
struct OneType {  // all levels of one type
  template <class F>
  static __device__ __forceinline__ void at(int, int, F&& f) {
    f(TypeC<TYPE>{});
  }
};
struct AnyType {  // two bits per level
  template <class F>
  static __device__ __forceinline__ void at(int types, int h, F&& f) {
    switch (types >> (2 * h) & 3) {
      case kUp: f(TypeC<kUp>{}); break;
      case kDown: f(TypeC<kDown>{}); break;
      case kSwap: f(TypeC<kSwap>{}); break;
      default: f(TypeC<kDrop>{}); break;
    }
  }
};

template <int KIND, int MODE, int K, class TY>
__device__ __forceinline__ void short_tile(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                           const float (&l)[kShortK], const float (&av)[kShortK],
                                           const float (&om)[kShortK], const float (&al)[kShortK], int lane) {
  constexpr bool REC = KIND == kFwdRec || KIND == kBwdRec;
  constexpr bool FWD = KIND == kFwd || KIND == kFwdRec;
  const int64_t sb = T.slot_base + lane;
  const bool real = lane < T.nbdd;
  const int ty = S.types;
  Costs<2> C[K + 1];  // the first pass' costs: SP(., T) or SP(r, .) of levels 0 .. K
  auto update = [&](int h, float b0, float b1) -> float {
    const float m0 = b0, m1 = l[h] + b1;
    const float Mn = __fmul_rn(MODE == 1 ? om[h] : a.omega0, m1 - m0);
    const float ln = unit_lambda_new<MODE>(l[h], Mn, al[h], av[h]);
    if (real) {
      a.lam[sb + h * kWarp] = ln;
      a.M[sb + h * kWarp] = Mn;
      if (REC) a.rec_diff[sb + h * kWarp] = m1 - m0;
    }
    return ln;
  };
  if (FWD) {
    C[K] = unit_end<2>(S.accept);
#pragma unroll
    for (int h = K - 1; h > 0; --h)
      TY::at(ty, h, [&](auto t) { C[h] = unit_up<2, decltype(t)::value>(C[h + 1], l[h]); });
    Costs<2> R = unit_root<2>(S.start);
#pragma unroll
    for (int h = 0; h < K; ++h)
      TY::at(ty, h, [&](auto t) {
        constexpr int TP = decltype(t)::value;
        float b0, b1;
        if (REC) {
          uint32_t rec = 0;
          unit_minima_rec<2, TP>(R, C[h + 1], b0, b1, rec);
          unit_up_rec<2, TP>(C[h + 1], l[h], rec);
          R = unit_down_rec<2, TP>(R, update(h, b0, b1), rec);
          if (real) a.rec_unit[sb + h * kWarp] = rec;
        } else {
          unit_minima<2, TP>(R, C[h + 1], b0, b1);
          R = unit_down<2, TP>(R, update(h, b0, b1));
        }
      });
  } else {
    C[0] = unit_root<2>(S.start);
#pragma unroll
    for (int h = 0; h < K - 1; ++h)
      TY::at(ty, h, [&](auto t) { C[h + 1] = unit_down<2, decltype(t)::value>(C[h], l[h]); });
    Costs<2> t2 = unit_end<2>(S.accept);
#pragma unroll
    for (int h = K - 1; h >= 0; --h)
      TY::at(ty, h, [&](auto t) {
        constexpr int TP = decltype(t)::value;
        float b0, b1;
        if (REC) {
          uint32_t rec = 0;
          unit_minima_rec<2, TP>(C[h], t2, b0, b1, rec);
          unit_down_rec<2, TP>(C[h], l[h], rec);
          t2 = unit_up_rec<2, TP>(t2, update(h, b0, b1), rec);
          if (real) a.rec_unit[sb + h * kWarp] = rec;
        } else {
          unit_minima<2, TP>(C[h], t2, b0, b1);
          t2 = unit_up<2, TP>(t2, update(h, b0, b1));
        }
      });
    if (a.E != nullptr && real) a.E[__ldg(A.slot_row + sb)] = S.start ? t2.v[1] : t2.v[0];
  }
}

template <int KIND, int MODE, int K>
__device__ __forceinline__ void short_types(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                            const float (&l)[kShortK], const float (&av)[kShortK],
                                            const float (&om)[kShortK], const float (&al)[kShortK], int lane) {
  if (S.nruns == 1 && (S.types & 3) == kUp)
    short_tile<KIND, MODE, K, OneType<kUp>>(A, a, T, S, l, av, om, al, lane);
  else if (S.nruns == 1 && (S.types & 3) == kDown)
    short_tile<KIND, MODE, K, OneType<kDown>>(A, a, T, S, l, av, om, al, lane);
  else
    short_tile<KIND, MODE, K, AnyType>(A, a, T, S, l, av, om, al, lane);
}

// One short tile.
template <int KIND, int MODE>
__device__ __forceinline__ void short_body(const DevArena& A, const SweepArgs& a, const Tile& T, const UnitShape& S,
                                           int lane) {
  const int64_t sb = T.slot_base + lane;
  const int k = T.nhops;
  int v[kShortK];
#pragma unroll
  for (int h = 0; h < kShortK; ++h) v[h] = h < k ? __ldcs(A.slot_var + sb + h * kWarp) : -1;
  grid_wait();
  grid_trigger();
  float l[kShortK], av[kShortK], om[kShortK], al[kShortK];
  const float* src = A.var_avg;
#pragma unroll
  for (int h = 0; h < kShortK; ++h) {
    const bool on = h < k;
    l[h] = on ? __ldcg(a.lam + sb + h * kWarp) : 0.0f;
    av[h] = v[h] >= 0 ? src[v[h]] : 0.0f;
    om[h] = MODE == 1 && on ? __ldcg(a.omega + sb + h * kWarp) : 0.0f;
    al[h] = MODE == 1 && on ? __ldcg(a.alpha + sb + h * kWarp) : 0.0f;
  }
  switch (k) {
    case 1: short_types<KIND, MODE, 1>(A, a, T, S, l, av, om, al, lane); break;
    case 2: short_types<KIND, MODE, 2>(A, a, T, S, l, av, om, al, lane); break;
    default: short_types<KIND, MODE, 3>(A, a, T, S, l, av, om, al, lane); break;
  }
}

template <int KIND, int MODE>
__global__ void __launch_bounds__(128) k_unit_short(DevArena A, SweepArgs a, int tile0, int tile1) {
  const int lane = threadIdx.x & 31;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (tile >= tile1) return;
  const Tile T = A.tiles[tile];
  short_body<KIND, MODE>(A, a, T, A.unit_shapes[T.unit - 1], lane);
}

template <int KIND, int MODE, int WMAX>
__global__ void __launch_bounds__(128) k_unit(DevArena A, SweepArgs a, int region_bytes, int tile0, int tile1) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + warp;
  if (tile >= tile1) return;  // whole warp leaves; no CTA-wide barrier follows
  constexpr bool UPDATE = KIND == kFwd || KIND == kBwd || KIND == kFwdRec || KIND == kBwdRec;
  constexpr int STRIDE = kStride<UPDATE, MODE>;
  const Tile T = A.tiles[tile];
  const int k = T.nhops;
  float* m = reinterpret_cast<float*>(smem + (size_t)warp * region_bytes);
  const uint64_t pol = l2_evict_first();
  // the variable ids come first, into the words of the averaging terms, so
  // that the gather can follow as soon as they are there: two memory latencies
  // per tile whatever its length (ids loaded into registers a few levels at a
  // time took one per few levels)
  if (UPDATE) {
    copy_rows<STRIDE>(m + kAvg, A.slot_var + T.slot_base, k, lane, pol);
    cp_async_commit();
  }
  const UnitShape S = A.unit_shapes[T.unit - 1];
  grid_wait();
  grid_trigger();
  copy_rows<STRIDE>(m, a.lam + T.slot_base, k, lane, pol);
  if (UPDATE && MODE == 1) {
    copy_rows<STRIDE>(m + kOm, a.omega + T.slot_base, k, lane, pol);
    copy_rows<STRIDE>(m + kAl, a.alpha + T.slot_base, k, lane, pol);
  }
  cp_async_commit();
  if (UPDATE) {
    cp_async_wait_one();
    __syncwarp();
    // the averaging terms (S_i in mode 1, S_i / |J_i| in mode 0) replace the
    // ids; they are not needed before the second pass
    const float* src = A.var_avg;
    float* q = m + kAvg + lane;
#pragma unroll 2
    for (int h = 0; h < k; ++h) {
      const int v = __float_as_int(*q);
      if (v >= 0) cp_async4(q, src + v);
      q += STRIDE;
    }
    cp_async_commit();
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

// ---- smoothed subproblems --------------------------------------------------
// E_a = -a log Z, Z = sum over feasible x of exp(<w, x>), w = -lambda / a, and
// the marginals P(x_i = 1): the walks of a forward sweep with sums of products
// in place of minima of sums.  A level's two weights 1 and exp(w) are divided
// by the larger (its logarithm joins log Z), so that they are 1 and
// exp(-|w|): one exponential per level and one fused multiply-add per arc,
// where sums in the logarithmic domain take an exponential and a logarithm per
// arc.  A product of weights is at least exp(-sum |w|) and a sum over paths at
// most 2^k, so with sum |w| <= 40 and k <= 60 nothing leaves the range of
// float32 (not the product of a prefix' and a suffix' sum either); a tile with
// a row beyond that takes the logarithmic walk.
struct SumProd {  // x: exp(-|w|), negative when w > 0 (the 0-arc then has it)
  template <int W>
  static __device__ __forceinline__ Costs<W> end(int accept) {
    Costs<W> c;
#pragma unroll
    for (int u = 0; u < W; ++u) c.v[u] = (accept >> u) & 1 ? 1.0f : 0.0f;
    return c;
  }
  static __device__ __forceinline__ float q0(float x) { return x < 0.0f ? -x : 1.0f; }
  static __device__ __forceinline__ float q1(float x) { return x < 0.0f ? 1.0f : x; }
  template <int W, int TYPE>
  static __device__ __forceinline__ Costs<W> up(const Costs<W>& T, float x) {
    const float a0 = q0(x), a1 = q1(x);
    Costs<W> r;
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int o = unit_o<TYPE>(u);
      r.v[u] = a0 * T.v[unit_z<TYPE>(u)];
      if (o >= 0 && o < W) r.v[u] = fmaf(a1, T.v[o], r.v[u]);
    }
    return r;
  }
  template <int W, int TYPE>
  static __device__ __forceinline__ Costs<W> down(const Costs<W>& F, float x) {
    const float a0 = q0(x), a1 = q1(x);
    Costs<W> r;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      float b = 0.0f;
#pragma unroll
      for (int u = 0; u < W; ++u) {
        if (unit_z<TYPE>(u) == w) b = fmaf(a0, F.v[u], b);
        if (unit_o<TYPE>(u) == w) b = fmaf(a1, F.v[u], b);
      }
      r.v[w] = b;
    }
    return r;
  }
  // the paths through the level's 1-arcs
  template <int W, int TYPE>
  static __device__ __forceinline__ float through(const Costs<W>& F, const Costs<W>& T, float x) {
    float s = 0.0f;
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int o = unit_o<TYPE>(u);
      if (o >= 0 && o < W) s = fmaf(F.v[u], T.v[o], s);
    }
    return q1(x) * s;
  }
  static __device__ __forceinline__ float share(float s, float Z) { return s / Z; }
};

// log(exp(x) + exp(y)) with -inf as the empty sum.
__device__ __forceinline__ float lse2(float x, float y) {
  const float m = fmaxf(x, y);
  if (m == -f_inf()) return m;
  return m + log1pf(expf(-fabsf(x - y)));
}

struct LogSum {  // x: w; everything a logarithm
  template <int W>
  static __device__ __forceinline__ Costs<W> end(int accept) {
    Costs<W> c;
#pragma unroll
    for (int u = 0; u < W; ++u) c.v[u] = (accept >> u) & 1 ? 0.0f : -f_inf();
    return c;
  }
  template <int W, int TYPE>
  static __device__ __forceinline__ Costs<W> up(const Costs<W>& T, float x) {
    Costs<W> r;
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int o = unit_o<TYPE>(u);
      r.v[u] = T.v[unit_z<TYPE>(u)];
      if (o >= 0 && o < W) r.v[u] = lse2(r.v[u], x + T.v[o]);
    }
    return r;
  }
  template <int W, int TYPE>
  static __device__ __forceinline__ Costs<W> down(const Costs<W>& F, float x) {
    Costs<W> r;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      float b = -f_inf();
#pragma unroll
      for (int u = 0; u < W; ++u) {
        if (unit_z<TYPE>(u) == w) b = lse2(b, F.v[u]);
        if (unit_o<TYPE>(u) == w) b = lse2(b, F.v[u] + x);
      }
      r.v[w] = b;
    }
    return r;
  }
  template <int W, int TYPE>
  static __device__ __forceinline__ float through(const Costs<W>& F, const Costs<W>& T, float x) {
    float s = -f_inf();
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int o = unit_o<TYPE>(u);
      if (o >= 0 && o < W) s = lse2(s, F.v[u] + x + T.v[o]);
    }
    return s;
  }
  static __device__ __forceinline__ float share(float s, float Z) { return expf(s - Z); }
};

template <class OP, int W>
__device__ __forceinline__ float smoothed_walk(const UnitCtx& s, int rows, const float* x0, float* cost, float* out,
                                               bool real, int lane) {
  const Costs<W> t = unit_first_up<W, kWarp, OP>(s, rows, x0, cost, lane);
  float Z = 0.0f;
#pragma unroll
  for (int u = 0; u < W; ++u)
    if (u == s.start) Z = t.v[u];
  Costs<W> F = OP::template end<W>(1 << s.start);
  unit_second_down<W, kWarp, OP>(s, x0, cost, lane, [&](auto ty, const float* x, const Costs<W>& t1) {
    constexpr int TY = decltype(ty)::value;
    const float m = OP::share(OP::template through<W, TY>(F, t1, x[0]), Z);
    if (real) *out = m;
    out += kWarp;
    F = OP::template down<W, TY>(F, x[0]);
  });
  return Z;
}

template <int W>
__device__ __forceinline__ void smoothed_tile(const DevArena& A, float a_s, float* E_a, float* marg, const Tile& T,
                                              const UnitShape& S, float* smem, int lane) {
  const UnitCtx s{S.k, S.start, S.accept, S.nruns, A.unit_runs + S.run_base};
  const int64_t sb = T.slot_base + lane;
  const bool real = lane < T.nbdd;
  float* x0 = smem + lane;
  float* cost = smem + s.k * kWarp;
  const float inv_a = 1.0f / a_s;
  float range = 0.0f;
  for (int h = 0; h < s.k; ++h) range += fabsf(x0[h * kWarp] * inv_a);
  // (not a number: out of range too)
  if (s.k <= 60 && __all_sync(0xffffffffu, !real || range <= 40.0f)) {
    float off = 0.0f, err = 0.0f;  // sum of the logarithms divided out, and its rounding (TwoSum)
    for (int h = 0; h < s.k; ++h) {
      const float w = -x0[h * kWarp] * inv_a;
      const float e = expf(-fabsf(w));
      x0[h * kWarp] = w > 0.0f ? -e : e;
      const float d = fmaxf(w, 0.0f), t = off + d, b = t - off;
      err += (off - (t - b)) + (d - b);
      off = t;
    }
    const float Z = smoothed_walk<SumProd, W>(s, S.rows, x0, cost, marg + sb, real, lane);
    if (E_a && real) E_a[__ldg(A.slot_row + sb)] = -a_s * (off + (err + logf(Z)));
  } else {
    for (int h = 0; h < s.k; ++h) x0[h * kWarp] = -x0[h * kWarp] * inv_a;
    const float Z = smoothed_walk<LogSum, W>(s, S.rows, x0, cost, marg + sb, real, lane);
    if (E_a && real) E_a[__ldg(A.slot_row + sb)] = -a_s * Z;
  }
}

template <int WMAX>
__global__ void __launch_bounds__(128) k_unit_smoothed(DevArena A, const float* lam, float a_s, float* E_a, float* marg,
                                                       int region_bytes, int tile0, int tile1) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + warp;
  if (tile >= tile1) return;  // whole warp leaves; no CTA-wide barrier follows
  const Tile T = A.tiles[tile];
  float* m = reinterpret_cast<float*>(smem + (size_t)warp * region_bytes);
  copy_rows<kWarp>(m, lam + T.slot_base, T.nhops, lane, l2_evict_first());
  cp_async_commit();
  const UnitShape S = A.unit_shapes[T.unit - 1];
  cp_async_wait_all();
  __syncwarp();
  if (S.W == 2)
    smoothed_tile<2>(A, a_s, E_a, marg, T, S, m, lane);
  else if (WMAX >= 4 && S.W == 4)
    smoothed_tile<4>(A, a_s, E_a, marg, T, S, m, lane);
  else if (WMAX >= 8 && S.W == 6)
    smoothed_tile<6>(A, a_s, E_a, marg, T, S, m, lane);
  else if (WMAX >= 8)
    smoothed_tile<8>(A, a_s, E_a, marg, T, S, m, lane);
}

// ---- adjoint of a recording sweep (see kernels_adjoint.cu) -----------------
// Per level and lane, staged: the gradient of lambda, the argmin word, m1 - m0,
// the averaging weight, {S-dot of the next sweep, S at the sweep's start} of
// the slot's variable (its id first, as in the sweeps), (mode 1) omega.
constexpr int kJRec = kWarp, kJDiff = 2 * kWarp, kJAl = 3 * kWarp, kJIn = 4 * kWarp, kJOm = 6 * kWarp;

template <int FWD, int MODE, int W>
__device__ __forceinline__ void unit_adjoint_tile(const AdjArgs& a, const Tile& T, const UnitCtx& s, float* smem,
                                                  int lane) {
  constexpr int STRIDE = kWarp * (MODE == 1 ? 7 : 6);
  const bool real = lane < T.nbdd;
  float* x = smem + lane + (FWD ? (s.k - 1) * STRIDE : 0);
  int64_t q = T.slot_base + lane + (FWD ? (s.k - 1) * kWarp : 0);
  // the update of a level reversed (g: gradient of lambda^new with the path
  // costs' share); returns the gradient d of m1 (that of m0 is -d).  The
  // running parameter gradients come through a ring of kAdjAhead levels, every
  // lane its own words (one level ahead in a register, each level cost the
  // latency of DRAM).
  const bool want_a = a.g_alpha != nullptr, want_w = a.g_omega != nullptr;
  float* ring = smem + s.k * STRIDE + lane;
  int p = 0;
  auto reverse = [&](float* y, float g) -> float {
    const int64_t at = q;
    q += FWD ? -kWarp : kWarp;
    cp_async_wait_but<kAdjAhead - 1>();
    float* r = ring + (p & (kAdjAhead - 1)) * 2 * kWarp;
    const float ca = r[0], cw = r[kWarp];
    __syncwarp();
    if (p + kAdjAhead < s.k) {
      const int64_t next = at + (FWD ? -kAdjAhead : kAdjAhead) * kWarp;
      if (want_a) cp_async4(r, a.g_alpha + next);
      if (want_w) cp_async4(r + kWarp, a.g_omega + next);
    }
    cp_async_commit();
    ++p;
    const float2 in = *reinterpret_cast<const float2*>(y - lane + kJIn + 2 * lane);
    const float seed = a.seed_M && real ? a.seed_M[at] : 0.0f;
    const float Mt = seed + in.x - g;
    const float d = (MODE == 1 ? y[kJOm] : a.omega0) * Mt;
    if (real) {
      a.sdot[at] = y[kJAl] * g;
      if (want_a) a.g_alpha[at] = ca + g * in.y;
      if (want_w) a.g_omega[at] = cw + Mt * y[kJDiff];
    }
    y[0] = g + d;
    y[kJDiff] = d;
    return d;
  };
  Costs<W> G;
#pragma unroll
  for (int u = 0; u < W; ++u) G.v[u] = 0.0f;
  if (FWD) {
    // SP(r, .) of level h + 1 was relaxed from level h with lambda^new_h
    unit_runs_up(s, [&](auto ty, int b, int e) {
      constexpr int TY = decltype(ty)::value;
      for (int n = e - b; n > 0; --n) {
        const uint32_t rec = __float_as_uint(x[kJRec]);
        float g = x[0];
        G = unit_route_in<W, TY>(G, rec, g);
        unit_seed_in<W>(G, rec, reverse(x, g));
        x -= STRIDE;
      }
    });
    // SP(., T) under lambda^old: its gradient flows top-down
    x += STRIDE;
#pragma unroll
    for (int u = 0; u < W; ++u) G.v[u] = 0.0f;
    unit_runs_down(s, [&](auto ty, int b, int e) {
      constexpr int TY = decltype(ty)::value;
      for (int n = e - b; n > 0; --n) {
        const uint32_t rec = __float_as_uint(x[kJRec]);
        float g = x[0];
        Costs<W> N;
#pragma unroll
        for (int u = 0; u < W; ++u) N.v[u] = 0.0f;
        unit_seed_out<W, TY>(N, rec, x[kJDiff]);
        unit_route_out<W, TY>(G, rec, N, g);
        G = N;
        x[0] = g;
        x += STRIDE;
      }
    });
  } else {
    // SP(., T) of level h was recomputed with lambda^new_h
    unit_runs_down(s, [&](auto ty, int b, int e) {
      constexpr int TY = decltype(ty)::value;
      for (int n = e - b; n > 0; --n) {
        const uint32_t rec = __float_as_uint(x[kJRec]);
        float g = x[0];
        Costs<W> N;
#pragma unroll
        for (int u = 0; u < W; ++u) N.v[u] = 0.0f;
        unit_route_out<W, TY>(G, rec, N, g);
        unit_seed_out<W, TY>(N, rec, reverse(x, g));
        G = N;
        x += STRIDE;
      }
    });
    // SP(r, .) under lambda^old: its gradient flows bottom-up
    x -= STRIDE;
#pragma unroll
    for (int u = 0; u < W; ++u) G.v[u] = 0.0f;
    unit_runs_up(s, [&](auto ty, int b, int e) {
      constexpr int TY = decltype(ty)::value;
      for (int n = e - b; n > 0; --n) {
        const uint32_t rec = __float_as_uint(x[kJRec]);
        float g = x[0];
        G = unit_route_in<W, TY>(G, rec, g);
        unit_seed_in<W>(G, rec, x[kJDiff]);
        x[0] = g;
        x -= STRIDE;
      }
    });
  }
  float* out = a.g_lam + T.slot_base + lane;
  x = smem + lane;
  if (real)
    for (int h = 0; h < s.k; ++h) out[h * kWarp] = x[h * STRIDE];
}

template <int FWD, int MODE, int WMAX>
__global__ void __launch_bounds__(128) k_unit_adjoint(DevArena A, AdjArgs a, int region_bytes, int tile0, int tile1) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int STRIDE = kWarp * (MODE == 1 ? 7 : 6);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = tile0 + blockIdx.x * (blockDim.x >> 5) + warp;
  if (tile >= tile1) return;  // whole warp leaves; no CTA-wide barrier follows
  const Tile T = A.tiles[tile];
  const int k = T.nhops;
  float* m = reinterpret_cast<float*>(smem + (size_t)warp * region_bytes);
  const uint64_t pol = l2_evict_first();
  copy_rows<STRIDE>(m + kJIn, A.slot_var + T.slot_base, k, lane, pol);
  cp_async_commit();
  const UnitShape S = A.unit_shapes[T.unit - 1];
  grid_wait();
  grid_trigger();
  copy_rows<STRIDE>(m, a.g_lam + T.slot_base, k, lane, pol);
  copy_rows<STRIDE>(m + kJRec, a.rec_unit + T.slot_base, k, lane, pol);
  copy_rows<STRIDE>(m + kJDiff, a.rec_diff + T.slot_base, k, lane, pol);
  copy_rows<STRIDE>(m + kJAl, (MODE == 1 ? a.alpha : A.slot_invdeg) + T.slot_base, k, lane, pol);
  if (MODE == 1) copy_rows<STRIDE>(m + kJOm, a.omega + T.slot_base, k, lane, pol);
  for (int j = 0; j < min(k, kAdjAhead); ++j) {  // the first levels of the ring
    const int64_t q = T.slot_base + lane + (FWD ? k - 1 - j : j) * kWarp;
    float* r = m + k * STRIDE + lane + j * 2 * kWarp;
    if (a.g_alpha) cp_async4(r, a.g_alpha + q);
    if (a.g_omega) cp_async4(r + kWarp, a.g_omega + q);
  }
  cp_async_commit();
  cp_async_wait_one();
  __syncwarp();
  for (int h = 0; h < k; ++h) {
    // the pairs replace the ids: every lane reads its id before any is overwritten
    float* in = m + h * STRIDE + kJIn;
    const int v = __float_as_int(in[lane]);
    __syncwarp();
    if (v >= 0) cp_async8(in + 2 * lane, a.var_in + v);
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncwarp();
  const UnitCtx s{S.k, S.start, S.accept, S.nruns, A.unit_runs + S.run_base};
  if (S.W == 2)
    unit_adjoint_tile<FWD, MODE, 2>(a, T, s, m, lane);
  else if (WMAX >= 4 && S.W == 4)
    unit_adjoint_tile<FWD, MODE, 4>(a, T, s, m, lane);
  else if (WMAX >= 8 && S.W == 6)
    unit_adjoint_tile<FWD, MODE, 6>(a, T, s, m, lane);
  else if (WMAX >= 8)
    unit_adjoint_tile<FWD, MODE, 8>(a, T, s, m, lane);
}

template <int FWD, int MODE>
void launch_adjoint_group(const DevArena& A, const AdjArgs& a, const AdjGroup& G, int wpc, size_t region, Chain& ch) {
  const int nt = G.tile1 - G.tile0, grid = (nt + wpc - 1) / wpc;
  auto k = G.unit_w <= 2 ? k_unit_adjoint<FWD, MODE, 2>
                         : (G.unit_w <= 4 ? k_unit_adjoint<FWD, MODE, 4> : k_unit_adjoint<FWD, MODE, 8>);
  chain_launch(ch, k, grid, wpc * kWarp, region * wpc, A, a, (int)region, G.tile0, G.tile1);
}

template <int FWD, int MODE>
cudaError_t set_adjoint_attr(int b) {
  cudaError_t e = cudaFuncSetAttribute(k_unit_adjoint<FWD, MODE, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_unit_adjoint<FWD, MODE, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_unit_adjoint<FWD, MODE, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  return e;
}

// ---- whole iterations of a small arena in one launch -----------------------
// An arena of a few unit tiles is latency alone: a sweep and a reduction are
// two launches of about 2 us each whatever they do.  One block instead keeps
// lambda, M and the per-variable sums in shared memory for the whole call; a
// block barrier stands between a sweep (a tile per warp at a time) and a
// reduction (a variable per thread), and the arrays go back at the end.  The
// operations and their order are the separate kernels'.
template <int MODE>
__global__ void __launch_bounds__(1024) k_small_iterate(DevArena A, SweepArgs a, int iters, int region_bytes) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int ns = (int)A.num_slots;
  float* lam = reinterpret_cast<float*>(smem);
  float* M = lam + ns;
  float* S = M + ns;
  float* row = reinterpret_cast<float*>(smem + ((size_t)(2 * ns + A.n) * 4 + 127) / 128 * 128 +
                                        (size_t)warp * region_bytes);
  constexpr int STRIDE = kStride<true, MODE>;
  grid_wait();
  grid_trigger();
  for (int q = threadIdx.x; q < ns; q += blockDim.x) {
    lam[q] = a.lam[q];
    M[q] = a.M[q];
  }
  __syncthreads();
  auto sum = [&](int i) {
    int q[kEll], b = 0, e = 0;
#pragma unroll
    for (int r = 0; r < kEll; ++r) q[r] = __ldg(A.var_ell + (int64_t)r * A.n + i);
    if (q[kEll - 1] <= -2) {
      q[kEll - 1] = -2 - q[kEll - 1];
      b = __ldg(A.var_ptr + i) + kEll;
      e = __ldg(A.var_ptr + i + 1);
    }
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < kEll; ++r)
      if (q[r] >= 0) s += M[q[r]];
    for (int k = b; k < e; ++k) s += M[__ldg(A.var_slots + k)];
    return s;
  };
  auto reduce = [&]() {
    for (int i = threadIdx.x; i < A.n; i += blockDim.x) {
      const float s = sum(i);
      S[i] = MODE == 1 ? s : __ldg(A.invdeg + i) * s;
    }
    __syncthreads();
  };
  SweepArgs w = a;
  w.lam = lam;
  w.M = M;
  auto sweep = [&](auto kind, float* E) {
    constexpr int KIND = decltype(kind)::value;
    w.E = E;
    for (int tile = warp; tile < A.num_tiles; tile += warps) {
      const Tile T = A.tiles[tile];
      const UnitShape sh = A.unit_shapes[T.unit - 1];
      const int64_t sb = T.slot_base + lane;
      float* x = row + lane;
      for (int h = 0; h < T.nhops; ++h) {
        const int64_t q = sb + h * kWarp;
        const int v = __ldg(A.slot_var + q);
        x[0] = lam[q];
        x[kAvg] = v >= 0 ? S[v] : 0.0f;
        if (MODE == 1) {
          x[kOm] = a.omega[q];
          x[kAl] = a.alpha[q];
        }
        x += STRIDE;
      }
      if (sh.W == 2)
        unit_tile<KIND, MODE, 2>(A, w, T, sh, row, lane);
      else if (sh.W == 4)
        unit_tile<KIND, MODE, 4>(A, w, T, sh, row, lane);
      else if (sh.W == 6)
        unit_tile<KIND, MODE, 6>(A, w, T, sh, row, lane);
      else
        unit_tile<KIND, MODE, 8>(A, w, T, sh, row, lane);
      __syncwarp();  // the next tile of another shape places its inputs over other lanes' path costs
    }
    __syncthreads();
  };
  for (int it = 0; it < iters; ++it) {
    reduce();
    sweep(TypeC<kFwd>{}, nullptr);
    reduce();
    sweep(TypeC<kBwd>{}, it + 1 == iters ? a.E : nullptr);
  }
  for (int q = threadIdx.x; q < ns; q += blockDim.x) {
    a.lam[q] = lam[q];
    a.M[q] = M[q];
  }
  for (int i = threadIdx.x; i < A.n; i += blockDim.x) {
    A.var_avg[i] = S[i];  // the last sweep's
    A.S[i] = sum(i);
  }
}

template <int KIND, int MODE>
void launch_group(const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region, Chain& ch) {
  const int nt = G.tile1 - G.tile0;
  if constexpr (KIND == kFwd || KIND == kBwd || KIND == kFwdRec || KIND == kBwdRec) {
    if (G.unit_short) {
      chain_launch(ch, k_unit_short<KIND, MODE>, (nt + 3) / 4, 128, 0, A, a, G.tile0, G.tile1);
      return;
    }
  }
  const int grid = (nt + wpc - 1) / wpc;
  auto k = G.unit_w <= 2 ? k_unit<KIND, MODE, 2> : (G.unit_w <= 4 ? k_unit<KIND, MODE, 4> : k_unit<KIND, MODE, 8>);
  chain_launch(ch, k, grid, wpc * kWarp, region * wpc, A, a, (int)region, G.tile0, G.tile1);
}

template <int KIND, int MODE>
cudaError_t set_attr(int b) {
  constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_unit<KIND, MODE, 2>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit<KIND, MODE, 4>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit<KIND, MODE, 8>, attr, b);
  return e;
}

}  // namespace

cudaError_t set_unit_smem_limit(size_t bytes) {
  const int b = (int)bytes;
  cudaError_t e = set_attr<kFwd, 0>(b);
  if (e == cudaSuccess) e = set_attr<kFwd, 1>(b);
  if (e == cudaSuccess) e = set_attr<kBwd, 0>(b);
  if (e == cudaSuccess) e = set_attr<kBwd, 1>(b);
  if (e == cudaSuccess) e = set_attr<kFwdRec, 0>(b);
  if (e == cudaSuccess) e = set_attr<kFwdRec, 1>(b);
  if (e == cudaSuccess) e = set_attr<kBwdRec, 0>(b);
  if (e == cudaSuccess) e = set_attr<kBwdRec, 1>(b);
  if (e == cudaSuccess) e = set_adjoint_attr<1, 0>(b);
  if (e == cudaSuccess) e = set_adjoint_attr<1, 1>(b);
  if (e == cudaSuccess) e = set_adjoint_attr<0, 0>(b);
  if (e == cudaSuccess) e = set_adjoint_attr<0, 1>(b);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_small_iterate<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_small_iterate<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit_smoothed<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit_smoothed<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_unit_smoothed<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  if (e == cudaSuccess) e = set_attr<kMinMarg, 0>(b);
  if (e == cudaSuccess) e = set_attr<kEnergy, 0>(b);
  if (e == cudaSuccess) e = set_attr<kSeed, 0>(b);
  return e;
}

void launch_unit(int kind, const DevArena& A, const SweepArgs& a, const LaunchGroup& G, int wpc, size_t region,
                 Chain& ch) {
  const bool m1 = a.mode == 1;
  switch (kind) {
    case kFwd: m1 ? launch_group<kFwd, 1>(A, a, G, wpc, region, ch) : launch_group<kFwd, 0>(A, a, G, wpc, region, ch); break;
    case kBwd: m1 ? launch_group<kBwd, 1>(A, a, G, wpc, region, ch) : launch_group<kBwd, 0>(A, a, G, wpc, region, ch); break;
    case kFwdRec:
      m1 ? launch_group<kFwdRec, 1>(A, a, G, wpc, region, ch) : launch_group<kFwdRec, 0>(A, a, G, wpc, region, ch);
      break;
    case kBwdRec:
      m1 ? launch_group<kBwdRec, 1>(A, a, G, wpc, region, ch) : launch_group<kBwdRec, 0>(A, a, G, wpc, region, ch);
      break;
    case kMinMarg: launch_group<kMinMarg, 0>(A, a, G, wpc, region, ch); break;
    case kEnergy: launch_group<kEnergy, 0>(A, a, G, wpc, region, ch); break;
    default: launch_group<kSeed, 0>(A, a, G, wpc, region, ch); break;
  }
}

namespace {
// lambda, M and the per-variable sums, and a warp's slice, in shared memory
size_t small_fixed(const DevArena& A) { return ((size_t)(2 * A.num_slots + A.n) * 4 + 127) / 128 * 128; }
size_t small_region(const LaunchGroup* groups, int num_groups, int mode) {
  size_t region = 0;
  for (int g = 0; g < num_groups; ++g)
    region = std::max(region, (size_t)(mode == 1 ? groups[g].unit_bytes1 : groups[g].unit_bytes0));
  return region;
}
int small_warps(const DevArena& A, size_t region, size_t smem_cap) {
  return (int)std::min<size_t>(std::min(32, A.num_tiles), (smem_cap - small_fixed(A)) / region);
}
}  // namespace

bool small_arena(const DevArena& A, const LaunchGroup* groups, int num_groups, size_t smem_cap) {
  if (A.unit_slots != A.num_slots || A.num_long > 0 || A.num_tiles < 1) return false;
  int64_t work = (int64_t)A.n + A.n / 5;
  for (int g = 0; g < num_groups; ++g) work += groups[g].work;
  if (work > kSmallWork) return false;
  const size_t region = small_region(groups, num_groups, 1);  // whatever the mode: the larger
  return small_fixed(A) + region <= smem_cap && small_warps(A, region, smem_cap) >= std::min(8, A.num_tiles);
}

bool launch_small_iterate(const DevArena& A, const SweepArgs& a, const LaunchGroup* groups, int num_groups, int iters,
                          size_t smem_cap, Chain& ch) {
  if (!small_arena(A, groups, num_groups, smem_cap)) return false;
  const size_t region = small_region(groups, num_groups, a.mode), fixed = small_fixed(A);
  const int warps = small_warps(A, region, smem_cap);
  // threads beyond the tiles' warps help the reduction
  const int threads = std::max(warps, std::min<int>(32, (A.n + 31) / 32)) * kWarp;
  const int blocks_warps = threads / kWarp;
  const size_t bytes = fixed + region * (size_t)blocks_warps;
  const int use = bytes <= smem_cap ? blocks_warps : warps;
  chain_launch(ch, a.mode == 1 ? k_small_iterate<1> : k_small_iterate<0>, 1, use * kWarp, fixed + region * use, A, a,
               iters, (int)region);
  return true;
}

void launch_unit_smoothed(const DevArena& A, const float* lam, float a_s, float* E_a, float* marg, const LaunchGroup& G,
                          int wpc, size_t region, cudaStream_t st) {
  const int nt = G.tile1 - G.tile0, grid = (nt + wpc - 1) / wpc;
  auto k = G.unit_w <= 2 ? k_unit_smoothed<2> : (G.unit_w <= 4 ? k_unit_smoothed<4> : k_unit_smoothed<8>);
  k<<<grid, wpc * kWarp, region * wpc, st>>>(A, lam, a_s, E_a, marg, (int)region, G.tile0, G.tile1);
}

void launch_unit_adjoint(bool forward, const DevArena& A, const AdjArgs& a, const AdjGroup& G, int wpc, size_t region,
                         Chain& ch) {
  if (forward)
    a.mode == 1 ? launch_adjoint_group<1, 1>(A, a, G, wpc, region, ch)
                : launch_adjoint_group<1, 0>(A, a, G, wpc, region, ch);
  else
    a.mode == 1 ? launch_adjoint_group<0, 1>(A, a, G, wpc, region, ch)
                : launch_adjoint_group<0, 0>(A, a, G, wpc, region, ch);
}

}  // namespace dg
