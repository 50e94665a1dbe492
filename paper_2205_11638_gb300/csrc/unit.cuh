// unit.cuh -- device building blocks of the unit tiles (UnitShape): one warp
// owns a tile of up to 32 BDDs of one shape, lane b owns BDD b, and a level's
// path costs are W registers of the lane.
//
// A unit row's BDD is a window of partial sums whose two arcs shift a state
// by at most one, so App. B's recursions need no child codes, no gathers and
// no per-node address arithmetic: SP(r, .) and SP(., T) of a level are W adds
// and W mins over registers, the state shifts are register names (the level
// type is the same for the whole warp), and only the costs of the direction
// opposite to the sweep go through shared memory (written by a first pass,
// one lane's own words, so without barriers).  Every cost is the value of the
// node-by-node kernels bit for bit: the same FP32 additions along the same
// arcs, and minima are exact in any order.
#pragma once

#include "sweep.cuh"

namespace dg {

// State reached from state u by the 0-arc / 1-arc of a level of type TYPE; -1
// and W are outside the window.
template <int TYPE>
__device__ __forceinline__ constexpr int unit_z(int u) {
  return TYPE == kSwap ? (u > 0 ? u - 1 : 0) : u;
}
template <int TYPE>
__device__ __forceinline__ constexpr int unit_o(int u) {
  return TYPE == kUp ? u + 1 : (TYPE == kSwap ? u : (TYPE == kDown ? (u > 0 ? u - 1 : 0) : u - 1));
}

template <int W>
struct Costs {
  float v[W];
  __device__ __forceinline__ float at(int u) const { return u >= 0 && u < W ? v[u] : f_inf(); }  // u is a constant
};

// Costs of a level from the costs T of the level below: SP(., T) of state u.
template <int W, int TYPE>
__device__ __forceinline__ Costs<W> unit_up(const Costs<W>& T, float l) {
  Costs<W> r;
#pragma unroll
  for (int u = 0; u < W; ++u) {
    const int o = unit_o<TYPE>(u);
    r.v[u] = T.at(unit_z<TYPE>(u));
    if (o >= 0 && o < W) r.v[u] = fminf(r.v[u], l + T.at(o));
  }
  return r;
}

// SP(r, .) of the next level from the costs R of a level.
template <int W, int TYPE>
__device__ __forceinline__ Costs<W> unit_down(const Costs<W>& R, float l) {
  Costs<W> r;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    float b = f_inf();
#pragma unroll
    for (int u = 0; u < W; ++u) {
      if (unit_z<TYPE>(u) == w) b = fminf(b, R.v[u]);
      if (unit_o<TYPE>(u) == w) b = fminf(b, R.v[u] + l);
    }
    r.v[w] = b;
  }
  return r;
}

// Minima over the level's states of SP(r, u) + SP(child, T) by the 0- and the
// 1-arc (as trees: a short chain between one level's update and the next).
template <int W, int TYPE>
__device__ __forceinline__ void unit_minima(const Costs<W>& R, const Costs<W>& T, float& b0, float& b1) {
  float x0[W], x1[W];
#pragma unroll
  for (int u = 0; u < W; ++u) {
    const int o = unit_o<TYPE>(u);
    x0[u] = R.v[u] + T.at(unit_z<TYPE>(u));
    x1[u] = o >= 0 && o < W ? R.v[u] + T.at(o) : f_inf();
  }
#pragma unroll
  for (int d = 1; d < W; d *= 2)
#pragma unroll
    for (int u = 0; u + d < W; u += 2 * d) {
      x0[u] = fminf(x0[u], x0[u + d]);
      x1[u] = fminf(x1[u], x1[u + d]);
    }
  b0 = x0[0];
  b1 = x1[0];
}

// Argmin records of one level of a recording sweep, one 32-bit word per slot:
//   bits 0..7    SP(state u, T) leaves u by its 1-arc
//   bits 8..16   in-arc of SP(r, w) on the next level: two bits for w = 0, one
//                for each other state, the index of the candidate in
//                unit_in_arc's order
//   bits 17..19  argmin state of m0, bits 20..22 of m1
// The candidates of a state are ordered as the tie rule wants them, by (parent
// rank, beta); ranks descend in the state number.
constexpr int kRecIn = 8, kRecV0 = 17, kRecV1 = 20;
__device__ __forceinline__ constexpr int unit_in_shift(int w) { return kRecIn + (w == 0 ? 0 : w + 1); }

// Calls f(candidate index, parent state, beta) for the arcs into state w.
template <int W, int TYPE, class F>
__device__ __forceinline__ void unit_in_arcs(int w, F&& f) {
  if (TYPE == kUp) {
    f(0, w, 0);
    if (w > 0) f(1, w - 1, 1);
  } else if (TYPE == kSwap) {
    if (w + 1 < W) f(0, w + 1, 0);
    f(1, w, w == 0 ? 0 : 1);
    if (w == 0) f(2, 0, 1);
  } else {
    if (w + 1 < W) f(0, w + 1, 1);
    f(1, w, 0);
    if (TYPE == kDown && w == 0) f(2, 0, 1);
  }
}

// unit_down that also records the in-arcs (the first strictly smallest
// candidate).
template <int W, int TYPE>
__device__ __forceinline__ Costs<W> unit_down_rec(const Costs<W>& R, float l, uint32_t& rec) {
  Costs<W> r;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    float b = f_inf();
    uint32_t c = 0;
    unit_in_arcs<W, TYPE>(w, [&](int i, int u, int beta) {
      const float x = beta ? R.v[u] + l : R.v[u];
      if (x < b) {
        b = x;
        c = (uint32_t)i << unit_in_shift(w);
      }
    });
    r.v[w] = b;
    rec |= c;
  }
  return r;
}

// unit_up that also records the out-arcs (the 0-arc on ties).
template <int W, int TYPE>
__device__ __forceinline__ Costs<W> unit_up_rec(const Costs<W>& T, float l, uint32_t& rec) {
  Costs<W> r;
#pragma unroll
  for (int u = 0; u < W; ++u) {
    const int o = unit_o<TYPE>(u);
    const float tl = T.at(unit_z<TYPE>(u));
    const float th = o >= 0 && o < W ? l + T.at(o) : f_inf();
    const bool take0 = tl <= th;
    r.v[u] = take0 ? tl : th;
    rec |= take0 ? 0u : 1u << u;
  }
  return r;
}

// unit_minima that also records the argmin states (the largest on ties).
template <int W, int TYPE>
__device__ __forceinline__ void unit_minima_rec(const Costs<W>& R, const Costs<W>& T, float& b0, float& b1,
                                                uint32_t& rec) {
  b0 = b1 = f_inf();
  uint32_t v0 = 0, v1 = 0;
#pragma unroll
  for (int u = W - 1; u >= 0; --u) {
    const int o = unit_o<TYPE>(u);
    const float x0 = R.v[u] + T.at(unit_z<TYPE>(u));
    if (x0 < b0) {
      b0 = x0;
      v0 = u;
    }
    if (o >= 0 && o < W) {
      const float x1 = R.v[u] + T.at(o);
      if (x1 < b1) {
        b1 = x1;
        v1 = u;
      }
    }
  }
  rec |= v0 << kRecV0 | v1 << kRecV1;
}

// Gradients G of SP(r, .) on the next level to the parents' level along the
// recorded in-arcs; g receives those that entered by a 1-arc.
template <int W, int TYPE>
__device__ __forceinline__ Costs<W> unit_route_in(const Costs<W>& G, uint32_t rec, float& g) {
  Costs<W> r;
#pragma unroll
  for (int u = 0; u < W; ++u) r.v[u] = 0.0f;
#pragma unroll
  for (int w = W - 1; w >= 0; --w) {
    const uint32_t c = rec >> unit_in_shift(w) & (w == 0 ? 3u : 1u);
    unit_in_arcs<W, TYPE>(w, [&](int i, int u, int beta) {
      const float x = c == (uint32_t)i ? G.v[w] : 0.0f;
      r.v[u] += x;
      if (beta) g += x;
    });
  }
  return r;
}

// Gradients G of SP(., T) of a level to the children's level (added to r)
// along the recorded out-arcs; g receives those that left by a 1-arc.
template <int W, int TYPE>
__device__ __forceinline__ void unit_route_out(const Costs<W>& G, uint32_t rec, Costs<W>& r, float& g) {
#pragma unroll
  for (int u = W - 1; u >= 0; --u) {
    const bool hi = (rec >> u) & 1u;
    const int z = unit_z<TYPE>(u), o = unit_o<TYPE>(u);
    r.v[z] += hi ? 0.0f : G.v[u];
    if (o >= 0 && o < W) {
      const float x = hi ? G.v[u] : 0.0f;
      r.v[o] += x;
      g += x;
    }
  }
}

// The gradients of the min-marginals (m1: d, m0: -d) at the argmin states:
// SP(r, .) of the level, SP(., T) of the children's level.
template <int W>
__device__ __forceinline__ void unit_seed_in(Costs<W>& r, uint32_t rec, float d) {
  const int v0 = (rec >> kRecV0) & 7u, v1 = (rec >> kRecV1) & 7u;
#pragma unroll
  for (int u = 0; u < W; ++u) {
    if (v0 == u) r.v[u] -= d;
    if (v1 == u) r.v[u] += d;
  }
}
template <int W, int TYPE>
__device__ __forceinline__ void unit_seed_out(Costs<W>& r, uint32_t rec, float d) {
  const int v0 = (rec >> kRecV0) & 7u, v1 = (rec >> kRecV1) & 7u;
#pragma unroll
  for (int u = 0; u < W; ++u) {
    const int o = unit_o<TYPE>(u);
    if (v0 == u) r.v[unit_z<TYPE>(u)] -= d;
    if (o >= 0 && o < W && v1 == u) r.v[o] += d;
  }
}

// The costs of a level in the warp's shared memory: 32 W floats per level,
// in pieces of four (or two) states per lane, so that a lane moves them with
// 16- (8-) byte accesses free of bank conflicts.
template <int W>
__device__ __forceinline__ void unit_store(float* row, const Costs<W>& c, int lane) {
  if constexpr (W % 4 == 0) {
#pragma unroll
    for (int j = 0; j < W / 4; ++j)
      reinterpret_cast<float4*>(row)[j * kWarp + lane] = make_float4(c.v[4 * j], c.v[4 * j + 1], c.v[4 * j + 2], c.v[4 * j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < W / 2; ++j)
      reinterpret_cast<float2*>(row)[j * kWarp + lane] = make_float2(c.v[2 * j], c.v[2 * j + 1]);
  }
}
template <int W>
__device__ __forceinline__ Costs<W> unit_load(const float* row, int lane) {
  Costs<W> c;
  if constexpr (W % 4 == 0) {
#pragma unroll
    for (int j = 0; j < W / 4; ++j) {
      const float4 x = reinterpret_cast<const float4*>(row)[j * kWarp + lane];
      c.v[4 * j] = x.x;
      c.v[4 * j + 1] = x.y;
      c.v[4 * j + 2] = x.z;
      c.v[4 * j + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < W / 2; ++j) {
      const float2 x = reinterpret_cast<const float2*>(row)[j * kWarp + lane];
      c.v[2 * j] = x.x;
      c.v[2 * j + 1] = x.y;
    }
  }
  return c;
}

// What the two-pass walks compute: path costs (minima of sums), or the sums
// over paths of the smoothed subproblems (kernels_unit.cu).
struct MinPlus {
  template <int W>
  static __device__ __forceinline__ Costs<W> end(int accept);
  template <int W, int TYPE>
  static __device__ __forceinline__ Costs<W> up(const Costs<W>& T, float l) {
    return unit_up<W, TYPE>(T, l);
  }
};

// SP(., T) below the last level, SP(r, .) of the first.
template <int W>
__device__ __forceinline__ Costs<W> unit_end(int accept) {
  Costs<W> c;
#pragma unroll
  for (int u = 0; u < W; ++u) c.v[u] = (accept >> u) & 1 ? 0.0f : f_inf();
  return c;
}
template <int W>
__device__ __forceinline__ Costs<W> unit_root(int start) {
  Costs<W> c;
#pragma unroll
  for (int u = 0; u < W; ++u) c.v[u] = u == start ? 0.0f : f_inf();
  return c;
}

template <int W>
__device__ __forceinline__ Costs<W> MinPlus::end(int accept) {
  return unit_end<W>(accept);
}

// One shape, as a warp holds it.
struct UnitCtx {
  int k, start, accept, nruns;
  const uint16_t* runs;
};

// Calls f(type constant, first level, end level) for the runs in ascending or
// descending order, so that a level's type is decided once per run.
template <int T>
struct TypeC {
  static constexpr int value = T;
};
template <class F>
__device__ __forceinline__ void unit_run(unsigned type, int b, int e, F& f) {
  switch (type) {
    case kUp: f(TypeC<kUp>{}, b, e); break;
    case kDown: f(TypeC<kDown>{}, b, e); break;
    case kSwap: f(TypeC<kSwap>{}, b, e); break;
    default: f(TypeC<kDrop>{}, b, e); break;
  }
}
template <class F>
__device__ __forceinline__ void unit_runs_down(const UnitCtx& s, F&& f) {
  int b = 0;
  for (int r = 0; r < s.nruns; ++r) {
    const unsigned run = __ldg(s.runs + r);
    unit_run(run & 3u, b, (int)(run >> 2), f);
    b = (int)(run >> 2);
  }
}
template <class F>
__device__ __forceinline__ void unit_runs_up(const UnitCtx& s, F&& f) {
  unsigned run = __ldg(s.runs + s.nruns - 1);
  for (int r = s.nruns - 1; r >= 0; --r) {
    const unsigned prev = r > 0 ? __ldg(s.runs + r - 1) : 0u;
    unit_run(run & 3u, (int)(prev >> 2), (int)(run >> 2), f);
    run = prev;
  }
}

// The two-pass walks.  The first pass leaves the costs of every second level
// of a run in shared memory, the second recomputes the others from their
// neighbour (the same operations on the same values) right before it needs
// them: half the shared memory per tile, which is what limits the warps per
// SM, for two operations per recomputed state.  x points at the lane's word of
// level 0 in the staged inputs (lambda first), STRIDE floats per level; the
// walks move pointers instead of indexing, because a level of a narrow row is
// only some twenty operations.

// First pass of a forward sweep: SP(., T) of the levels at even distance from
// their run's first level and of every run's end, in level order; returns those
// of level 0.
template <int W, int STRIDE, class OP = MinPlus>
__device__ __forceinline__ Costs<W> unit_first_up(const UnitCtx& s, int rows, const float* x, float* cost, int lane) {
  Costs<W> t = OP::template end<W>(s.accept);
  float* p = cost + rows * (kWarp * W);
  x += s.k * STRIDE;
  unit_runs_up(s, [&](auto ty, int b, int e) {
    constexpr int TY = decltype(ty)::value;
    if (e < s.k) unit_store<W>(p -= kWarp * W, t, lane);
    int n = e - b;
    if (n & 1) {
      x -= STRIDE;
      t = OP::template up<W, TY>(t, x[0]);
      if (--n > 0) unit_store<W>(p -= kWarp * W, t, lane);
    }
    for (; n > 0; n -= 2) {
      t = OP::template up<W, TY>(t, x[-STRIDE]);
      x -= 2 * STRIDE;
      t = OP::template up<W, TY>(t, x[0]);
      if (n > 2) unit_store<W>(p -= kWarp * W, t, lane);
    }
  });
  return t;
}
// Second pass: f(type constant, x of level h, SP(., T) of level h + 1) for
// every level in ascending order.
template <int W, int STRIDE, class OP = MinPlus, class F>
__device__ __forceinline__ void unit_second_down(const UnitCtx& s, const float* x, const float* cost, int lane,
                                                 F&& f) {
  const float* p = cost;
  unit_runs_down(s, [&](auto ty, int b, int e) {
    constexpr int TY = decltype(ty)::value;
    const int last = e == s.k ? 2 : 0;  // levels left when SP(., T) of the next stored level is the terminals'
    int n = e - b;
    for (; n >= 2; n -= 2) {
      Costs<W> t2 = OP::template end<W>(s.accept);
      if (n != last) {
        t2 = unit_load<W>(p, lane);
        p += kWarp * W;
      }
      const Costs<W> t1 = OP::template up<W, TY>(t2, x[STRIDE]);
      f(ty, x, t1);
      f(ty, x + STRIDE, t2);
      x += 2 * STRIDE;
    }
    if (n > 0) {
      Costs<W> t1 = OP::template end<W>(s.accept);
      if (last == 0) {
        t1 = unit_load<W>(p, lane);
        p += kWarp * W;
      }
      f(ty, x, t1);
      x += STRIDE;
    }
  });
}

// The same for a backward sweep: SP(r, .) of the levels at even distance from
// their run's first level, then f(type constant, x of level h, SP(r, .) of
// level h) in descending order.
template <int W, int STRIDE>
__device__ __forceinline__ void unit_first_down(const UnitCtx& s, const float* x, float* cost, int lane) {
  Costs<W> R = unit_root<W>(s.start);
  float* p = cost;
  unit_runs_down(s, [&](auto ty, int b, int e) {
    constexpr int TY = decltype(ty)::value;
    int n = e - b;
    for (bool stored = b > 0; n > 0; n -= 2, stored = true) {
      if (stored) {
        unit_store<W>(p, R, lane);
        p += kWarp * W;
      }
      R = unit_down<W, TY>(R, x[0]);
      if (n > 1) R = unit_down<W, TY>(R, x[STRIDE]);
      x += (n > 1 ? 2 : 1) * STRIDE;
    }
  });
}
template <int W, int STRIDE, class F>
__device__ __forceinline__ void unit_second_up(const UnitCtx& s, int rows, const float* x, const float* cost,
                                               int lane, F&& f) {
  const float* p = cost + rows * (kWarp * W);
  x += s.k * STRIDE;
  unit_runs_up(s, [&](auto ty, int b, int e) {
    constexpr int TY = decltype(ty)::value;
    const int first = b == 0 ? 2 : 0;  // levels left when SP(r, .) of the run's first level is the root's
    int n = e - b;
    if (n & 1) {
      Costs<W> r0 = unit_root<W>(s.start);
      if (n != 1 || b > 0) r0 = unit_load<W>(p -= kWarp * W, lane);
      x -= STRIDE;
      f(ty, x, r0);
      --n;
    }
    for (; n > 0; n -= 2) {
      Costs<W> r0 = unit_root<W>(s.start);
      if (n != first) r0 = unit_load<W>(p -= kWarp * W, lane);
      x -= 2 * STRIDE;
      const Costs<W> r1 = unit_down<W, TY>(r0, x[0]);
      f(ty, x + STRIDE, r1);
      f(ty, x, r0);
    }
  });
}

// lambda^new of the update, every rounding spelled out as the mixed tiles'
// kernel has it: M^new = omega (m1 - m0) rounded on its own, the mode-1 term
// alpha S by one fused multiply-add.
template <int MODE>
__device__ __forceinline__ float unit_lambda_new(float l, float Mn, float al, float av) {
  const float r = l - Mn;
  return MODE == 1 ? __fmaf_rn(al, av, r) : r + av;
}

// Asynchronous 4-byte global -> shared copy (a gather: every lane its own
// address), through L1.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
template <int N>  // all but the last N groups
__device__ __forceinline__ void cp_async_wait_but() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace dg
