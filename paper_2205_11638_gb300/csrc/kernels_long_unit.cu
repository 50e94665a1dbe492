// kernels_long_unit.cu -- the long unit rows (LongItem): long cardinality and
// assignment rows, whose BDDs are too large for a tile lane but have at most
// 32 states a level that two shifts connect (see UnitShape).
//
// The levels of one BDD are a chain (the paper's long subproblems: the update
// of a level needs the path costs under the lambda of the level before), so a
// sweep's time is the levels times the latency of one step, and everything
// else has to be out of that chain.  Up to 8 states a level are one lane's
// registers, as in the unit tiles: a step is some twenty instructions on a
// short chain, and the BDDs are spread thinly over the warps, since a warp that
// is alone on its scheduler waits for every instruction.  Wider levels are held
// by a segment of G lanes, lane s its state s: a step is one shuffle to the
// neighbour state, the segment's minima and the update.  All inputs of a work item are staged in shared
// memory before the walk (asynchronous copies; the averaging terms gathered
// through the staged variable ids), the costs opposite to the sweep are
// recomputed into shared memory by a first walk, and each step's words are
// read one step ahead.  New lambda and M replace the staged inputs and leave
// in one coalesced pass.  The loops over explicit children and in-arcs in
// global memory (kernels_long.cu) take half a microsecond a level, but need no
// shared memory: long, wide and many rows make their plain sweeps there (see
// where Plan::long_plain is set).
//
// Same FP32 operations, tie rules and records as there: results are equal bit
// for bit, gradients up to the rounding of sums.
#include "kernels.h"
#include "unit.cuh"

namespace dg {

namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;

// The segment of a lane.
template <int G>
struct LSeg {
  int base, s;
  int row;  // its BDD, among the item's
};

template <int G>
__device__ __forceinline__ float seg_min(float x) {
  if constexpr (G == 32) {
    // one reduction instead of five shuffles, over an order-preserving map
    const int i = __float_as_int(x);
    const int m = __reduce_min_sync(kAll, i ^ ((i >> 31) & 0x7FFFFFFF));
    return __int_as_float(m ^ ((m >> 31) & 0x7FFFFFFF));
  } else {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(kAll, x, o));
    return x;
  }
}
template <int G>
__device__ __forceinline__ float seg_sum(float x) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kAll, x, o);
  return x;
}
template <int G>
__device__ __forceinline__ uint32_t seg_bits(bool p, int base) {
  return (__ballot_sync(kAll, p) >> base) & (G == 32 ? kAll : (1u << (G & 31)) - 1u);
}

template <int G, int TYPE>
__device__ __forceinline__ int lz(int s) {
  return TYPE == kSwap ? max(s - 1, 0) : s;
}
template <int G, int TYPE>
__device__ __forceinline__ int lo_(int s) {  // may be -1 or G: no such state
  return TYPE == kUp ? s + 1 : (TYPE == kSwap ? s : (TYPE == kDown ? max(s - 1, 0) : s - 1));
}

// Value of the neighbour state the arcs come from (down) or lead to (up), inf
// outside the window.
template <int G, int TYPE>
__device__ __forceinline__ float from_neighbour(float R, const LSeg<G>& g, float none) {
  const int n = TYPE == kUp ? g.s - 1 : g.s + 1;
  const float x = __shfl_sync(kAll, R, g.base + (n & (G - 1)));
  return n >= 0 && n < G ? x : none;
}

// SP(., T) of the two children of the lane's state, from the level below.
template <int G, int TYPE>
__device__ __forceinline__ void children(float t, const LSeg<G>& g, float& tz, float& to) {
  const int n = TYPE == kUp ? g.s + 1 : g.s - 1;
  float x = __shfl_sync(kAll, t, g.base + (n & (G - 1)));
  if (TYPE == kDown || TYPE == kSwap) x = n < 0 ? t : x;  // the lowest state absorbs
  else x = n >= 0 && n < G ? x : f_inf();
  tz = TYPE == kSwap ? x : t;
  to = TYPE == kSwap ? t : x;
}

// SP(r, .) of the lane's state on the next level.
template <int G, int TYPE>
__device__ __forceinline__ float down(float R, float n, float l, int s) {
  if (TYPE == kSwap) return fminf(s == 0 ? fminf(R, R + l) : R + l, n);
  const float r = fminf(R, n + l);
  return TYPE == kDown && s == 0 ? fminf(r, R + l) : r;
}
// ... with the index of the in-arc in unit_in_arcs' order.
template <int G, int TYPE>
__device__ __forceinline__ float down_rec(float R, float n, float l, int s, int& c) {
  float x0, x1, x2 = f_inf();
  if (TYPE == kUp) {
    x0 = R;
    x1 = n + l;
  } else if (TYPE == kSwap) {
    x0 = n;
    x1 = s == 0 ? R : R + l;
    if (s == 0) x2 = R + l;
  } else {
    x0 = n + l;
    x1 = R;
    if (TYPE == kDown && s == 0) x2 = R + l;
  }
  float b = f_inf();
  c = 0;
  if (x0 < b) b = x0;
  if (x1 < b) {
    b = x1;
    c = 1;
  }
  if (x2 < b) {
    b = x2;
    c = 2;
  }
  return b;
}

// Runs of one level type over [0, kmax): the last run ends there.
template <class F>
__device__ __forceinline__ void runs_down(const DevArena& A, const LongItem& it, F&& f) {
  int b = 0;
  for (int r = 0; r < it.nruns; ++r) {
    const unsigned run = __ldg(A.unit_runs + it.run_base + r);
    const int e = r + 1 < it.nruns ? (int)(run >> 2) : it.kmax;
    unit_run(run & 3u, b, e, f);
    b = e;
  }
}
template <class F>
__device__ __forceinline__ void runs_up(const DevArena& A, const LongItem& it, F&& f) {
  int e = it.kmax;
  for (int r = it.nruns - 1; r >= 0; --r) {
    const unsigned run = __ldg(A.unit_runs + it.run_base + r);
    const int b = r > 0 ? (int)(__ldg(A.unit_runs + it.run_base + r - 1) >> 2) : 0;
    unit_run(run & 3u, b, e, f);
    e = b;
  }
}

// k floats (whole 16-byte pieces; slot ranges are padded to 32) to shared memory.
__device__ __forceinline__ void copy_row(float* dst, const void* src, int k, int lane, uint64_t pol) {
  for (int p = lane; p < (k + 3) / 4; p += kWarp) cp_async16(dst + 4 * p, (const char*)src + 16 * p, pol);
}

// The walk of a sweep with a level's states on the lanes of a segment: lam and
// avg (the staged inputs) receive the new lambda and M (kMinMarg: m1 and m0,
// kSeed: the minimising assignment in avg).  Segments beyond the item's BDDs
// repeat another one (same addresses, same values); steps are guarded only
// past the shortest BDD's levels (kmin).  Reads one level ahead may go one
// level past either end: the arrays have that much room.
template <int KIND, int MODE, int G>
__device__ __forceinline__ void walk_segments(const DevArena& A, const SweepArgs& a, const LongItem& it, float* lam,
                                              float* avg, const float* om, const float* al, float* cost, int lane) {
  constexpr bool REC = KIND == kFwdRec || KIND == kBwdRec;
  constexpr bool FWD = KIND == kFwd || KIND == kFwdRec;
  constexpr bool BWD = KIND == kBwd || KIND == kBwdRec;
  const int ST = long_unit_stride(it.kmax), TS = it.nseg * G;
  LSeg<G> g;
  g.s = lane & (G - 1);
  g.base = lane - g.s;
  g.row = (lane / G) % it.nseg;
  const LongBdd B = A.longs[A.long_order[it.first + g.row]];
  const int k = B.k, kmin = __reduce_min_sync(kAll, k);
  float* ml = lam + g.row * ST;
  float* ma = avg + g.row * ST;
  const float* mo = om + g.row * ST;
  const float* mw = al + g.row * ST;
  float* mt = cost + g.row * G + g.s;  // level h at mt[h TS], the terminals' at level k
  const float end = (it.accept >> g.s) & 1u ? 0.0f : f_inf();
  const float root = g.s == it.start ? 0.0f : f_inf();
  auto down_levels = [&](auto&& step) {
    runs_down(A, it, [&](auto ty, int b, int e) {
      const int m = min(e, kmin);
      int h = b;
      for (; h < m; ++h) step(ty, h, true);
      for (; h < e; ++h) step(ty, h, h < k);
    });
  };
  auto up_levels = [&](auto&& step) {
    runs_up(A, it, [&](auto ty, int b, int e) {
      const int m = max(b, kmin);
      int h = e - 1;
      for (; h >= m; --h) step(ty, h, h < k);
      for (; h >= b; --h) step(ty, h, true);
    });
  };
  struct In {  // a level's inputs
    float l, av, w, al;
  };
  auto input = [&](int h) {
    return In{ml[h], ma[h], MODE == 1 ? mo[h] : a.omega0, MODE == 1 ? mw[h] : 0.0f};
  };
  auto first_up = [&]() -> float {  // SP(., T) of every level; returns level 0's
    float t = end;
    mt[k * TS] = end;
    float l = ml[it.kmax - 1];
    up_levels([&](auto ty, int h, bool on) {
      const float l1 = ml[h - 1];
      float tz, to;
      children<G, decltype(ty)::value>(t, g, tz, to);
      if (on) {
        t = fminf(tz, l + to);
        mt[h * TS] = t;
      }
      l = l1;
    });
    return t;
  };
  // the update of a level from its minima, by every lane of the segment
  auto update = [&](int h, const In& x, bool on, float b0, float b1) -> float {
    const float m0 = b0, m1 = x.l + b1;
    const float Mn = __fmul_rn(x.w, m1 - m0);
    const float ln = unit_lambda_new<MODE>(x.l, Mn, x.al, x.av);
    if (g.s == 0 && on) {
      ml[h] = ln;
      ma[h] = Mn;
      if (REC) a.rec_diff[(int64_t)B.slot_base + h] = m1 - m0;
    }
    return ln;
  };
  auto record = [&](int h, bool on, bool hi, int c, float x0, float m0, float x1, float m1) {
    const uint32_t tb = seg_bits<G>(hi, g.base), rb = seg_bits<G>((c & 1) != 0, g.base);
    const uint32_t ex = seg_bits<G>(c == 2, g.base) & 1u;
    // the argmins: the largest state on ties
    const uint32_t b0 = seg_bits<G>(x0 == m0, g.base), b1 = seg_bits<G>(x1 == m1, g.base);
    const int v0 = b0 ? 31 - __clz((int)b0) : 0, v1 = b1 ? 31 - __clz((int)b1) : 0;
    if (g.s == 0 && on)
      reinterpret_cast<uint4*>(a.rec_lunit)[(int64_t)B.slot_base + h - A.long_slot_base] =
          make_uint4(tb, rb, (uint32_t)v0 | (uint32_t)v1 << 8 | ex << 16, 0u);
  };

  if (FWD || KIND == kMinMarg) {
    first_up();
    __syncwarp();
    float R = root;
    In in = input(0);
    runs_down(A, it, [&](auto ty, int b, int e) {
      constexpr int TY = decltype(ty)::value;
      const int oi = lo_<G, TY>(g.s);
      const bool ov = oi >= 0 && oi < G;
      const float* pz = mt + lz<G, TY>(g.s) - g.s;
      const float* po = mt + (ov ? oi : g.s) - g.s;
      float tz = pz[(b + 1) * TS], to = po[(b + 1) * TS];
      auto step = [&](int h, bool on) {
        const In nxt = input(h + 1);
        const float tz1 = pz[(h + 2) * TS], to1 = po[(h + 2) * TS];
        __syncwarp();  // every lane has read a level before any replaces its inputs
        const float n = from_neighbour<G, TY>(R, g, f_inf());
        const float x0 = R + tz, x1 = ov ? R + to : f_inf();
        const float b0 = seg_min<G>(x0), b1 = seg_min<G>(x1);
        if (KIND == kMinMarg) {
          if (g.s == 0 && on) {
            ml[h] = in.l + b1;
            ma[h] = b0;
          }
          R = down<G, TY>(R, n, in.l, g.s);
        } else {
          const float ln = update(h, in, on, b0, b1);
          if (REC) {
            int c;
            const bool hi = !(tz <= (ov ? in.l + to : f_inf()));
            R = down_rec<G, TY>(R, n, ln, g.s, c);
            record(h, on, hi, c, x0, b0, x1, b1);
          } else {
            R = down<G, TY>(R, n, ln, g.s);
          }
        }
        in = nxt;
        tz = tz1;
        to = to1;
      };
      const int m = min(e, kmin);
      int h = b;
      for (; h < m; ++h) step(h, true);
      for (; h < e; ++h) step(h, h < k);
    });
  } else if (BWD) {
    {
      float R = root;
      float l = ml[0];
      down_levels([&](auto ty, int h, bool on) {
        constexpr int TY = decltype(ty)::value;
        const float l1 = ml[h + 1];
        if (on) mt[h * TS] = R;
        R = down<G, TY>(R, from_neighbour<G, TY>(R, g, f_inf()), l, g.s);
        l = l1;
      });
    }
    __syncwarp();
    float t = end;
    In in = input(it.kmax - 1);
    float r = mt[(it.kmax - 1) * TS];
    up_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const In nxt = input(h - 1);
      const float r1 = mt[max(h - 1, 0) * TS];
      __syncwarp();  // as above
      float tz, to;
      children<G, TY>(t, g, tz, to);
      const float x0 = r + tz, x1 = r + to;
      const float b0 = seg_min<G>(x0), b1 = seg_min<G>(x1);
      const float ln = update(h, in, on, b0, b1);
      const float th = ln + to;
      if (REC) {
        constexpr int ni = TY == kUp ? -1 : 1;
        const bool nv = g.s + ni >= 0 && g.s + ni < G;
        int c;
        down_rec<G, TY>(r, nv ? mt[h * TS + ni] : f_inf(), in.l, g.s, c);
        const bool hi = !(tz <= th);
        record(h, on, hi, c, x0, b0, x1, b1);
        if (on) t = hi ? th : tz;
      } else if (on) {
        t = fminf(tz, th);
      }
      in = nxt;
      r = r1;
    });
    if (a.E != nullptr && g.s == it.start) a.E[B.row] = t;  // E^j = SP(r, T)
  } else {
    const float t = first_up();
    if (KIND == kEnergy) {
      if (a.E != nullptr && g.s == it.start) a.E[B.row] = t;
    } else {
      // kSeed: walk the minimising path from the root, the 0-arc on ties
      __syncwarp();
      int at = it.start;
      const float* row = cost + g.row * G;
      down_levels([&](auto ty, int h, bool on) {
        constexpr int TY = decltype(ty)::value;
        if (!on) return;
        const int z = lz<G, TY>(at), o = lo_<G, TY>(at);
        const float* p = row + (h + 1) * TS;
        const float c0 = p[z], c1 = o >= 0 && o < G ? p[o] : f_inf();
        // an infinite cost is the bottom terminal (the path stays feasible)
        const bool take0 = c0 < f_inf() && (c1 == f_inf() || c0 <= ml[h] + c1);
        if (g.s == 0) ma[h] = take0 ? 0.f : 1.f;
        at = take0 ? z : max(min(o, G - 1), 0);
      });
    }
  }
}

// ... with a level's states in the registers of the BDD's lane.  Lanes beyond
// the item's BDDs repeat another lane's (same addresses, same values), so that
// nothing diverges; only past the shortest BDD's levels (kmin) are the steps
// guarded.  Reads one level ahead may go one level past either end: the arrays
// have that much room.
template <int KIND, int MODE, int W>
__device__ __forceinline__ void walk_lanes(const DevArena& A, const SweepArgs& a, const LongItem& it, float* lam,
                                           float* avg, const float* om, const float* al, float* cost, int lane) {
  constexpr bool REC = KIND == kFwdRec || KIND == kBwdRec;
  constexpr bool FWD = KIND == kFwd || KIND == kFwdRec;
  constexpr bool BWD = KIND == kBwd || KIND == kBwdRec;
  const int ST = long_unit_stride(it.kmax), row = lane % it.nseg, TS = it.nseg * W;
  const LongBdd B = A.longs[A.long_order[it.first + row]];
  const int k = B.k, kmin = __reduce_min_sync(kAll, k);
  float* ml = lam + row * ST;
  float* ma = avg + row * ST;
  const float* mo = om + row * ST;
  const float* mw = al + row * ST;
  float* mt = cost + row * W;  // level h at mt[h TS], the terminals' at level k
  auto put = [&](int h, const Costs<W>& c) {
    if constexpr (W == 2) {
      *reinterpret_cast<float2*>(mt + h * TS) = make_float2(c.v[0], c.v[1]);
    } else {
#pragma unroll
      for (int j = 0; j < W / 4; ++j)
        reinterpret_cast<float4*>(mt + h * TS)[j] = make_float4(c.v[4 * j], c.v[4 * j + 1], c.v[4 * j + 2], c.v[4 * j + 3]);
    }
  };
  auto get = [&](int h) {
    Costs<W> c;
    if constexpr (W == 2) {
      const float2 x = *reinterpret_cast<const float2*>(mt + h * TS);
      c.v[0] = x.x;
      c.v[1] = x.y;
    } else {
#pragma unroll
      for (int j = 0; j < W / 4; ++j) {
        const float4 x = reinterpret_cast<const float4*>(mt + h * TS)[j];
        c.v[4 * j] = x.x;
        c.v[4 * j + 1] = x.y;
        c.v[4 * j + 2] = x.z;
        c.v[4 * j + 3] = x.w;
      }
    }
    return c;
  };
  const Costs<W> end = unit_end<W>((int)it.accept);
  const Costs<W> root = unit_root<W>(it.start);
  struct In {  // a level's inputs
    float l, av, w, al;
  };
  auto input = [&](int h) {
    return In{ml[h], ma[h], MODE == 1 ? mo[h] : a.omega0, MODE == 1 ? mw[h] : 0.0f};
  };
  // step(type, level) for the levels in ascending / descending order, of a BDD
  // shorter than the level none
  auto down_levels = [&](auto&& step) {
    runs_down(A, it, [&](auto ty, int b, int e) {
      const int m = min(e, kmin);
      int h = b;
#pragma unroll 2
      for (; h < m; ++h) step(ty, h, true);
      for (; h < e; ++h) step(ty, h, h < k);
    });
  };
  auto up_levels = [&](auto&& step) {
    runs_up(A, it, [&](auto ty, int b, int e) {
      const int m = max(b, kmin);
      int h = e - 1;
      for (; h >= m; --h) step(ty, h, h < k);
#pragma unroll 2
      for (; h >= b; --h) step(ty, h, true);
    });
  };
  auto first_up = [&]() {
    Costs<W> t = end;
    put(k, end);
    float l = ml[it.kmax - 1];
    up_levels([&](auto ty, int h, bool on) {
      const float l1 = ml[h - 1];
      if (on) {
        t = unit_up<W, decltype(ty)::value>(t, l);
        put(h, t);
      }
      l = l1;
    });
    return t;
  };
  auto update = [&](int h, const In& x, float b0, float b1) -> float {
    const float m0 = b0, m1 = x.l + b1;
    const float Mn = __fmul_rn(x.w, m1 - m0);
    const float ln = unit_lambda_new<MODE>(x.l, Mn, x.al, x.av);
    ml[h] = ln;
    ma[h] = Mn;
    if (REC) a.rec_diff[(int64_t)B.slot_base + h] = m1 - m0;
    return ln;
  };
  auto energy = [&](const Costs<W>& t) {  // E^j = SP(r, T)
    if (a.E == nullptr) return;
    float e = f_inf();
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (u == it.start) e = t.v[u];
    a.E[B.row] = e;
  };
  const int words = A.long_rec_words;
  uint32_t* rec_out = REC ? a.rec_lunit + (int64_t)(B.slot_base - A.long_slot_base) * words : nullptr;

  if (FWD || KIND == kMinMarg) {
    first_up();
    __syncwarp();
    Costs<W> R = root;
    In in = input(0);
    Costs<W> t1 = get(1);
    down_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const In nxt = input(h + 1);
      const Costs<W> t2 = get(h + 2);
      __syncwarp();
      if (on) {
        float b0, b1;
        if (REC) {
          uint32_t rec = 0;
          unit_minima_rec<W, TY>(R, t1, b0, b1, rec);
          unit_up_rec<W, TY>(t1, in.l, rec);
          R = unit_down_rec<W, TY>(R, update(h, in, b0, b1), rec);
          rec_out[h * words] = rec;
        } else {
          unit_minima<W, TY>(R, t1, b0, b1);
          float ln = in.l;
          if (KIND == kMinMarg) {
            ml[h] = in.l + b1;
            ma[h] = b0;
          } else {
            ln = update(h, in, b0, b1);
          }
          R = unit_down<W, TY>(R, ln);
        }
      }
      in = nxt;
      t1 = t2;
    });
  } else if (BWD) {
    {
      Costs<W> R = root;
      float l = ml[0];
      down_levels([&](auto ty, int h, bool on) {
        const float l1 = ml[h + 1];
        if (on) {
          put(h, R);
          R = unit_down<W, decltype(ty)::value>(R, l);
        }
        l = l1;
      });
    }
    __syncwarp();
    Costs<W> t = end;
    In in = input(it.kmax - 1);
    Costs<W> r = get(it.kmax - 1);
    up_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const In nxt = input(h - 1);
      const Costs<W> r1 = get(max(h - 1, 0));
      __syncwarp();
      if (on) {
        float b0, b1;
        if (REC) {
          uint32_t rec = 0;
          unit_minima_rec<W, TY>(r, t, b0, b1, rec);
          unit_down_rec<W, TY>(r, in.l, rec);
          t = unit_up_rec<W, TY>(t, update(h, in, b0, b1), rec);
          rec_out[h * words] = rec;
        } else {
          unit_minima<W, TY>(r, t, b0, b1);
          t = unit_up<W, TY>(t, update(h, in, b0, b1));
        }
      }
      in = nxt;
      r = r1;
    });
    energy(t);
  } else {
    const Costs<W> t = first_up();
    if (KIND == kEnergy) {
      energy(t);
    } else {
      // kSeed: walk the minimising path from the root, the 0-arc on ties
      __syncwarp();
      int at = it.start;
      down_levels([&](auto ty, int h, bool on) {
        constexpr int TY = decltype(ty)::value;
        if (!on) return;
        const int z = lz<W, TY>(at), o = lo_<W, TY>(at);
        const float* p = mt + (h + 1) * TS;
        const float c0 = p[z], c1 = o >= 0 && o < W ? p[o] : f_inf();
        // an infinite cost is the bottom terminal (the path stays feasible)
        const bool take0 = c0 < f_inf() && (c1 == f_inf() || c0 <= ml[h] + c1);
        ma[h] = take0 ? 0.f : 1.f;
        at = take0 ? z : max(min(o, W - 1), 0);
      });
    }
  }
}

template <int KIND, int MODE, int G>
__device__ __forceinline__ void long_unit_item(const DevArena& A, const SweepArgs& a, const LongItem& it, float* smem,
                                               int lane) {
  constexpr bool UPDATE = KIND == kFwd || KIND == kBwd || KIND == kFwdRec || KIND == kBwdRec;
  const int ST = long_unit_stride(it.kmax), nrow = it.nseg * ST;
  float* lam = smem + 4;  // room for the level before the first
  float* avg = lam + nrow;
  float* om = avg + nrow;
  float* al = om + (MODE == 1 ? nrow : 0);
  float* cost = al + (MODE == 1 ? nrow : 0);

  // ---- staging -------------------------------------------------------------
  const uint64_t pol = l2_evict_first();
  if (UPDATE) {
    for (int r = 0; r < it.nseg; ++r) {
      const LongBdd B = A.longs[A.long_order[it.first + r]];
      copy_row(avg + r * ST, A.slot_var + B.slot_base, B.k, lane, pol);
    }
    cp_async_commit();
  }
  grid_wait();
  grid_trigger();
  for (int r = 0; r < it.nseg; ++r) {
    const LongBdd B = A.longs[A.long_order[it.first + r]];
    copy_row(lam + r * ST, a.lam + B.slot_base, B.k, lane, pol);
    if (UPDATE && MODE == 1) {
      copy_row(om + r * ST, a.omega + B.slot_base, B.k, lane, pol);
      copy_row(al + r * ST, a.alpha + B.slot_base, B.k, lane, pol);
    }
  }
  cp_async_commit();
  if (UPDATE) {
    cp_async_wait_one();
    __syncwarp();
    const float* src = A.var_avg;
    for (int r = 0; r < it.nseg; ++r) {
      const int k = A.longs[A.long_order[it.first + r]].k;
#pragma unroll 4
      for (int h = lane; h < k; h += kWarp) {
        const int v = __float_as_int(avg[r * ST + h]);
        cp_async4(avg + r * ST + h, src + v);
      }
    }
    cp_async_commit();
  }
  cp_async_wait_all();
  __syncwarp();

  // ---- the walk --------------------------------------------------------------
  if constexpr (G <= kUnitMaxW)
    walk_lanes<KIND, MODE, G>(A, a, it, lam, avg, om, al, cost, lane);
  else
    walk_segments<KIND, MODE, G>(A, a, it, lam, avg, om, al, cost, lane);

  // ---- the new state ---------------------------------------------------------
  if (KIND == kEnergy) return;
  __syncwarp();
  for (int r = 0; r < it.nseg; ++r) {
    const LongBdd Br = A.longs[A.long_order[it.first + r]];
    float* o0 = (KIND == kMinMarg ? a.out2 : a.lam) + Br.slot_base;
    float* o1 = a.M + Br.slot_base;
    for (int h = lane; h < Br.k; h += kWarp) {
      if (KIND != kSeed) o0[h] = lam[r * ST + h];
      o1[h] = avg[r * ST + h];
    }
  }
}

template <int KIND, int MODE>
__global__ void __launch_bounds__(32) k_long_unit(DevArena A, SweepArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x;
  const LongItem it = A.long_items[blockIdx.x];
  float* p = reinterpret_cast<float*>(smem);
  switch (it.G) {
    case 2: long_unit_item<KIND, MODE, 2>(A, a, it, p, lane); break;
    case 4: long_unit_item<KIND, MODE, 4>(A, a, it, p, lane); break;
    case 8: long_unit_item<KIND, MODE, 8>(A, a, it, p, lane); break;
    case 16: long_unit_item<KIND, MODE, 16>(A, a, it, p, lane); break;
    default: long_unit_item<KIND, MODE, 32>(A, a, it, p, lane); break;
  }
}

// The reverse walk with the gradients of a level's path costs on the lanes of
// a segment.  Replaces, per level, the gradient of lambda^new by lambda^old's
// (gl), the weight by the contribution to S-dot (al), and the pair by the
// contributions to omega-dot and alpha-dot (in).
template <int FWD, int MODE, int G>
__device__ __forceinline__ void adjoint_segments(const DevArena& A, const AdjArgs& a, const LongItem& it,
                                                 const uint4* rec, float2* in, float* gl, float* df, float* al,
                                                 const float* om, int lane) {
  const int ST = long_unit_stride(it.kmax);
  LSeg<G> g;
  g.s = lane & (G - 1);
  g.base = lane - g.s;
  const bool act = lane / G < it.nseg;
  g.row = act ? lane / G : 0;
  const LongBdd B = A.longs[A.long_order[it.first + g.row]];
  const int k = B.k;
  const bool own = act && g.s == 0;
  float* mg = gl + g.row * ST;
  float* md = df + g.row * ST;
  float* mw = al + g.row * ST;
  const float* mo = om + g.row * ST;
  float2* mi = in + g.row * ST;
  const uint4* mr = rec + g.row * ST;
  const float* seed = a.seed_M ? a.seed_M + B.slot_base : nullptr;

  // the update of level h reversed (on: the BDD has that level, else nothing is
  // written and the result is not used); returns the gradient of m1
  auto reverse = [&](int h, bool on, float gs) -> float {
    h = min(h, k - 1);
    const float x = mg[h] + gs;
    const float2 v = mi[h];
    const float Mt = (seed ? seed[h] : 0.0f) + v.x - x;
    const float d = (MODE == 1 ? mo[h] : a.omega0) * Mt;
    __syncwarp();
    if (own && on) {
      mi[h] = make_float2(Mt * md[h], x * v.y);  // omega-dot, alpha-dot
      mw[h] = mw[h] * x;                         // contribution to S-dot
      md[h] = d;
      mg[h] = x + d;
    }
    return d;
  };
  // gradient of SP(r, .) from level h + 1 to level h; gs: what entered by 1-arcs
  auto route_in = [&](auto ty, float G2, const uint4& w, float& gs) -> float {
    constexpr int TY = decltype(ty)::value;
    const int c = (int)((w.y >> g.s) & 1u) | (g.s == 0 ? (int)((w.z >> 16) & 1u) << 1 : 0);
    float stay, moved, hi;
    if (TY == kUp) {
      stay = c == 0 ? G2 : 0.0f;
      moved = hi = c == 1 ? G2 : 0.0f;
    } else {
      moved = c == 0 ? G2 : 0.0f;
      stay = c != 0 ? G2 : 0.0f;
      hi = TY == kSwap ? (c == (g.s == 0 ? 2 : 1) ? G2 : 0.0f) : (c != 1 ? G2 : 0.0f);
    }
    const int n = TY == kUp ? g.s + 1 : g.s - 1;
    const float x = __shfl_sync(kAll, moved, g.base + (n & (G - 1)));
    gs = seg_sum<G>(hi);
    return stay + (n >= 0 && n < G ? x : 0.0f);
  };
  // gradient of SP(., T) from level h to level h + 1; gs: what left by 1-arcs
  auto route_out = [&](auto ty, float G1, const uint4& w, float& gs) -> float {
    constexpr int TY = decltype(ty)::value;
    const bool hi = (w.x >> g.s) & 1u;
    const float hp = hi ? G1 : 0.0f, lp = hi ? 0.0f : G1;
    const float moved = TY == kSwap ? lp : hp;
    float r = TY == kSwap ? hp : lp;
    const int n = TY == kUp ? g.s - 1 : g.s + 1;
    const float x = __shfl_sync(kAll, moved, g.base + (n & (G - 1)));
    if (n >= 0 && n < G) r += x;
    if ((TY == kDown || TY == kSwap) && g.s == 0) r += moved;  // the lowest state absorbs
    gs = seg_sum<G>(hp);
    return r;
  };
  auto seed_in = [&](float x, const uint4& w, float d) {
    if (g.s == (int)(w.z & 255u)) x -= d;
    if (g.s == (int)(w.z >> 8 & 255u)) x += d;
    return x;
  };
  auto seed_out = [&](auto ty, float x, const uint4& w, float d) {
    constexpr int TY = decltype(ty)::value;
    if (g.s == lz<G, TY>((int)(w.z & 255u))) x -= d;
    if (g.s == lo_<G, TY>((int)(w.z >> 8 & 255u))) x += d;
    return x;
  };
  const uint4 none = make_uint4(0u, 0u, 0u, 0u);
  float x = 0.0f;
  if (FWD) {
    // SP(r, .) of level h + 1 was relaxed from level h with lambda^new_h
    runs_up(A, it, [&](auto ty, int b, int e) {
      for (int h = e - 1; h >= b; --h) {
        const bool on = h < k;
        const uint4 w = on ? mr[h] : none;
        float gs;
        const float y = route_in(ty, x, w, gs);
        const float d = reverse(h, on, gs);
        x = on ? seed_in(y, w, d) : 0.0f;
      }
    });
  } else {
    // SP(., T) of level h was recomputed with lambda^new_h
    runs_down(A, it, [&](auto ty, int b, int e) {
      for (int h = b; h < e; ++h) {
        const bool on = h < k;
        const uint4 w = on ? mr[h] : none;
        float gs;
        const float y = route_out(ty, x, w, gs);
        const float d = reverse(h, on, gs);
        x = on ? seed_out(ty, y, w, d) : 0.0f;
      }
    });
  }
  __syncwarp();
  x = 0.0f;
  if (FWD) {
    // SP(., T) under lambda^old: its gradient flows top-down
    runs_down(A, it, [&](auto ty, int b, int e) {
      for (int h = b; h < e; ++h) {
        const bool on = h < k;
        const uint4 w = on ? mr[h] : none;
        float gs;
        const float y = route_out(ty, x, w, gs);
        x = seed_out(ty, y, w, on ? md[h] : 0.0f);
        if (own && on) mg[h] += gs;
      }
    });
  } else {
    // SP(r, .) under lambda^old: its gradient flows bottom-up
    runs_up(A, it, [&](auto ty, int b, int e) {
      for (int h = e - 1; h >= b; --h) {
        const bool on = h < k;
        const uint4 w = on ? mr[h] : none;
        float gs;
        const float y = route_in(ty, x, w, gs);
        x = on ? seed_in(y, w, md[h]) : 0.0f;
        if (own && on) mg[h] += gs;
      }
    });
  }
}

// ... in the registers of the BDD's lane (lanes and levels as in walk_lanes).
template <int FWD, int MODE, int W>
__device__ __forceinline__ void adjoint_lanes(const DevArena& A, const AdjArgs& a, const LongItem& it,
                                              const uint32_t* rec, float2* in, float* gl, float* df, float* al,
                                              const float* om, int lane) {
  const int ST = long_unit_stride(it.kmax), row = lane % it.nseg;
  const LongBdd B = A.longs[A.long_order[it.first + row]];
  const int k = B.k, kmin = __reduce_min_sync(kAll, k), last = k - 1;
  float* mg = gl + row * ST;
  float* md = df + row * ST;
  float* mw = al + row * ST;
  const float* mo = om + row * ST;
  float2* mi = in + row * ST;
  const uint32_t* mr = rec + row * ST;
  const float* seed = a.seed_M ? a.seed_M + B.slot_base : nullptr;
  auto down_levels = [&](auto&& step) {
    runs_down(A, it, [&](auto ty, int b, int e) {
      const int m = min(e, kmin);
      int h = b;
      for (; h < m; ++h) step(ty, h, true);
      for (; h < e; ++h) step(ty, h, h < k);
    });
  };
  auto up_levels = [&](auto&& step) {
    runs_up(A, it, [&](auto ty, int b, int e) {
      const int m = max(b, kmin);
      int h = e - 1;
      for (; h >= m; --h) step(ty, h, h < k);
      for (; h >= b; --h) step(ty, h, true);
    });
  };
  struct In {  // a level's inputs, read one level ahead
    uint32_t rec;
    float g, df, w, om, seed;
    float2 v;
  };
  auto input = [&](int h) {
    const int x = min(max(h, 0), last);
    return In{mr[x], mg[x], md[x], mw[x], MODE == 1 ? mo[x] : a.omega0, seed ? seed[x] : 0.0f, mi[x]};
  };
  auto reverse = [&](int h, const In& x, float g) -> float {
    const float Mt = x.seed + x.v.x - g;
    const float d = x.om * Mt;
    mi[h] = make_float2(Mt * x.df, g * x.v.y);
    mw[h] = x.w * g;
    md[h] = d;
    mg[h] = g + d;
    return d;
  };
  Costs<W> x;
  auto clear = [&](Costs<W>& c) {
#pragma unroll
    for (int u = 0; u < W; ++u) c.v[u] = 0.0f;
  };
  clear(x);
  if (FWD) {
    // SP(r, .) of level h + 1 was relaxed from level h with lambda^new_h
    In v = input(it.kmax - 1);
    up_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const In nxt = input(h - 1);
      __syncwarp();
      if (on) {
        float g = v.g;
        x = unit_route_in<W, TY>(x, v.rec, g);
        unit_seed_in<W>(x, v.rec, reverse(h, v, g));
      }
      v = nxt;
    });
    __syncwarp();
    // SP(., T) under lambda^old: its gradient flows top-down
    clear(x);
    uint32_t rc = mr[0];
    float d = md[0], g0 = mg[0];
    down_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const int n = min(h + 1, last);
      const uint32_t rc1 = mr[n];
      const float d1 = md[n], g1 = mg[n];
      __syncwarp();
      if (on) {
        Costs<W> y;
        clear(y);
        float g = 0.0f;
        unit_seed_out<W, TY>(y, rc, d);
        unit_route_out<W, TY>(x, rc, y, g);
        x = y;
        mg[h] = g0 + g;
        rc = rc1;
        d = d1;
        g0 = g1;
      }
    });
  } else {
    // SP(., T) of level h was recomputed with lambda^new_h
    In v = input(0);
    down_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const In nxt = input(h + 1);
      __syncwarp();
      if (on) {
        Costs<W> y;
        clear(y);
        float g = v.g;
        unit_route_out<W, TY>(x, v.rec, y, g);
        unit_seed_out<W, TY>(y, v.rec, reverse(h, v, g));
        x = y;
      }
      v = nxt;
    });
    __syncwarp();
    // SP(r, .) under lambda^old: its gradient flows bottom-up
    clear(x);
    uint32_t rc = mr[last];
    float d = md[last], g0 = mg[last];
    up_levels([&](auto ty, int h, bool on) {
      constexpr int TY = decltype(ty)::value;
      const int n = max(h - 1, 0);
      const uint32_t rc1 = mr[n];
      const float d1 = md[n], g1 = mg[n];
      __syncwarp();
      if (on) {
        float g = 0.0f;
        x = unit_route_in<W, TY>(x, rc, g);
        unit_seed_in<W>(x, rc, d);
        mg[h] = g0 + g;
        rc = rc1;
        d = d1;
        g0 = g1;
      }
    });
  }
}

// Adjoint of a recording sweep: the reverse of the walk with the gradients of
// a level's path costs on the segment's lanes (see kernels_adjoint.cu for the
// steps and kernels_unit.cu for the routing along the recorded arcs).
template <int FWD, int MODE, int G>
__device__ __forceinline__ void long_unit_adjoint_item(const DevArena& A, const AdjArgs& a, const LongItem& it,
                                                       float* smem, int lane) {
  const int ST = long_unit_stride(it.kmax), nrow = it.nseg * ST;
  uint4* rec = reinterpret_cast<uint4*>(smem);
  float2* in = reinterpret_cast<float2*>(rec + nrow);
  float* gl = reinterpret_cast<float*>(in + nrow);
  float* df = gl + nrow;
  float* al = df + nrow;
  float* om = al + nrow;
  float* id = om + nrow;
  const uint64_t pol = l2_evict_first();
  for (int r = 0; r < it.nseg; ++r) {
    const LongBdd B = A.longs[A.long_order[it.first + r]];
    copy_row(id + r * ST, A.slot_var + B.slot_base, B.k, lane, pol);
  }
  cp_async_commit();
  grid_wait();
  grid_trigger();
  for (int r = 0; r < it.nseg; ++r) {
    const LongBdd B = A.longs[A.long_order[it.first + r]];
    copy_row(gl + r * ST, a.g_lam + B.slot_base, B.k, lane, pol);
    copy_row(df + r * ST, a.rec_diff + B.slot_base, B.k, lane, pol);
    copy_row(al + r * ST, (MODE == 1 ? a.alpha : A.slot_invdeg) + B.slot_base, B.k, lane, pol);
    if (MODE == 1) copy_row(om + r * ST, a.omega + B.slot_base, B.k, lane, pol);
    // (a lane's BDD: the first word of a slot, side by side)
    const int words = A.long_rec_words;
    const uint32_t* src = a.rec_lunit + (int64_t)(B.slot_base - A.long_slot_base) * words;
    if (G > kUnitMaxW)
      for (int h = lane; h < B.k; h += kWarp) cp_async16(rec + r * ST + h, src + 4 * h, pol);
    else if (words == 1)
      copy_row(reinterpret_cast<float*>(rec) + r * ST, src, B.k, lane, pol);
    else
      for (int h = lane; h < B.k; h += kWarp) cp_async4(reinterpret_cast<uint32_t*>(rec) + r * ST + h, src + 4 * h);
  }
  cp_async_commit();
  cp_async_wait_one();
  __syncwarp();
  for (int r = 0; r < it.nseg; ++r) {
    const int k = A.longs[A.long_order[it.first + r]].k;
#pragma unroll 4
    for (int h = lane; h < k; h += kWarp) cp_async8(in + r * ST + h, a.var_in + __float_as_int(id[r * ST + h]));
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncwarp();

  if constexpr (G <= kUnitMaxW)
    adjoint_lanes<FWD, MODE, G>(A, a, it, reinterpret_cast<const uint32_t*>(rec), in, gl, df, al, om, lane);
  else
    adjoint_segments<FWD, MODE, G>(A, a, it, rec, in, gl, df, al, om, lane);
  __syncwarp();
  for (int r = 0; r < it.nseg; ++r) {
    const LongBdd Br = A.longs[A.long_order[it.first + r]];
    const int64_t q = Br.slot_base;
    for (int h = lane; h < Br.k; h += kWarp) {
      const float2 v = in[r * ST + h];
      a.sdot[q + h] = al[r * ST + h];
      a.g_lam[q + h] = gl[r * ST + h];
      if (a.g_omega) a.g_omega[q + h] += v.x;
      if (a.g_alpha) a.g_alpha[q + h] += v.y;
    }
  }
}

template <int FWD, int MODE>
__global__ void __launch_bounds__(32) k_long_unit_adjoint(DevArena A, AdjArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x;
  const LongItem it = A.long_items[blockIdx.x];
  float* p = reinterpret_cast<float*>(smem);
  switch (it.G) {
    case 2: long_unit_adjoint_item<FWD, MODE, 2>(A, a, it, p, lane); break;
    case 4: long_unit_adjoint_item<FWD, MODE, 4>(A, a, it, p, lane); break;
    case 8: long_unit_adjoint_item<FWD, MODE, 8>(A, a, it, p, lane); break;
    case 16: long_unit_adjoint_item<FWD, MODE, 16>(A, a, it, p, lane); break;
    default: long_unit_adjoint_item<FWD, MODE, 32>(A, a, it, p, lane); break;
  }
}

template <int KIND>
void launch_kind(const DevArena& A, const SweepArgs& a, Chain& ch) {
  chain_launch(ch, a.mode == 1 ? k_long_unit<KIND, 1> : k_long_unit<KIND, 0>, A.num_long_items, kWarp,
               A.long_unit_smem[a.mode == 1], A, a);
}

}  // namespace

cudaError_t set_long_unit_smem_limit(size_t bytes) {
  const int b = (int)bytes;
  constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_long_unit<kFwd, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kFwd, 1>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kBwd, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kBwd, 1>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kFwdRec, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kFwdRec, 1>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kBwdRec, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kBwdRec, 1>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kMinMarg, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kEnergy, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit<kSeed, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit_adjoint<0, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit_adjoint<0, 1>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit_adjoint<1, 0>, attr, b);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_unit_adjoint<1, 1>, attr, b);
  return e;
}

void launch_long_unit(int kind, const DevArena& A, const SweepArgs& a, Chain& ch) {
  switch (kind) {
    case kFwd: launch_kind<kFwd>(A, a, ch); break;
    case kBwd: launch_kind<kBwd>(A, a, ch); break;
    case kFwdRec: launch_kind<kFwdRec>(A, a, ch); break;
    case kBwdRec: launch_kind<kBwdRec>(A, a, ch); break;
    case kMinMarg: chain_launch(ch, k_long_unit<kMinMarg, 0>, A.num_long_items, kWarp, A.long_unit_smem[0], A, a); break;
    case kEnergy: chain_launch(ch, k_long_unit<kEnergy, 0>, A.num_long_items, kWarp, A.long_unit_smem[0], A, a); break;
    default: chain_launch(ch, k_long_unit<kSeed, 0>, A.num_long_items, kWarp, A.long_unit_smem[0], A, a); break;
  }
}

void launch_long_unit_adjoint(bool forward, const DevArena& A, const AdjArgs& a, Chain& ch) {
  auto k = forward ? (a.mode == 1 ? k_long_unit_adjoint<1, 1> : k_long_unit_adjoint<1, 0>)
                   : (a.mode == 1 ? k_long_unit_adjoint<0, 1> : k_long_unit_adjoint<0, 0>);
  chain_launch(ch, k, A.num_long_items, kWarp, A.long_unit_adj_smem, A, a);
}

}  // namespace dg
