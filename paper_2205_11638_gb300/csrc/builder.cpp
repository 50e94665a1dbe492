// builder.cpp -- host side of dg_plan: rows -> canonical quasi-reduced BDDs
// -> tiles -> the structure-of-arrays image of the device arena.
//
// BDDs (App. B of DOGE-Train): one per constraint row; level h holds the nodes
// of the row's h-th variable (ascending variable id), every root-to-top path
// meets one node per level and the paths are exactly the feasible
// assignments.  A node is identified with the set of feasible completions of
// the partial sums that reach it; nodes of a level are ordered by
// (lo rank, hi rank) with bottom = -2 < top = -1 < ranks, so that the
// minimal quasi-reduced BDD of a row is one fixed table.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <numeric>
#include <string>
#include <thread>
#include <unordered_map>

#include "dg_internal.h"

namespace dg {

namespace {

constexpr int kCodeBot = -2;
constexpr int kCodeTop = -1;
constexpr size_t kMaxStatesPerRow = size_t(1) << 22;

struct RowResult {
  int status = 0;  // dg_status
  std::string msg;
};

// Scratch reused across the rows one host thread builds.
struct RowScratch {
  std::vector<int64_t> sums;      // reachable partial sums (clamped), level by level
  std::vector<int64_t> rem_lo, rem_hi;  // per level: least / largest sum of the remaining terms
  std::vector<size_t> lvl;        // level offsets into sums
  std::vector<int32_t> code;      // code of every (level, sum)
  std::vector<uint64_t> keys;     // (lo+2) << 32 | (hi+2) per sum of a level
  std::vector<std::vector<uint64_t>> level_keys;  // per level: its nodes' keys, ascending
  int64_t nodes = 0;
  int maxw = 0;
};

inline bool row_holds(int64_t act, int sense, int64_t rhs) {
  switch (sense) {
    case 0: return act <= rhs;
    case 1: return act >= rhs;
    default: return act == rhs;
  }
}

inline int key_lo(uint64_t key) { return int(key >> 32) - 2; }
inline int key_hi(uint64_t key) { return int(key & 0xFFFFFFFFu) - 2; }

// Builds the BDD of one row: on success sc.level_keys[h] holds the nodes of
// level h in canonical order as keys (lo code + 2) << 32 | (hi code + 2),
// codes being ranks on level h + 1 with bottom = -2 and top = -1.
RowResult build_row(const int32_t* a, int k, int sense, int64_t rhs, RowScratch& sc) {
  RowResult res;
  // 1. partial sums reachable from the root, per level (sorted, unique).  A
  // partial sum s of level g behaves like any other sum outside the window
  // [rhs - rem_hi[g] - 1, rhs - rem_lo[g] + 1] on the same side of it (below
  // it every completion is feasible for '<=' and none for '>=' and '='; above
  // it the reverse), and adding a term keeps it outside, so sums are clamped
  // to the window: the same residual functions, hence the same BDD, from
  // O(k * window) partial sums instead of every reachable one.
  sc.rem_lo.assign(k + 1, 0);
  sc.rem_hi.assign(k + 1, 0);
  for (int h = k - 1; h >= 0; --h) {
    sc.rem_lo[h] = sc.rem_lo[h + 1] + std::min<int64_t>(0, a[h]);
    sc.rem_hi[h] = sc.rem_hi[h + 1] + std::max<int64_t>(0, a[h]);
  }
  auto clamp = [&](int64_t v, int g) {
    return std::min(std::max(v, rhs - sc.rem_hi[g] - 1), rhs - sc.rem_lo[g] + 1);
  };
  sc.sums.clear();
  sc.lvl.assign(1, 0);
  sc.sums.push_back(clamp(0, 0));
  sc.lvl.push_back(1);
  for (int h = 0; h < k; ++h) {
    size_t b = sc.lvl[h], e = sc.lvl[h + 1];
    size_t p = b, q = b;
    while (p < e || q < e) {  // merge {s} and {s + a_h}, both ascending (clamping is monotone)
      int64_t x = p < e ? clamp(sc.sums[p], h + 1) : INT64_MAX;
      int64_t y = q < e ? clamp(sc.sums[q] + a[h], h + 1) : INT64_MAX;
      int64_t v = std::min(x, y);
      if (x == v) ++p;
      if (y == v) ++q;
      if (sc.sums.size() == e || sc.sums.back() != v) sc.sums.push_back(v);
    }
    sc.lvl.push_back(sc.sums.size());
    if (sc.sums.size() > kMaxStatesPerRow) {
      res.status = DG_EINVAL;
      res.msg = "row has too many distinct partial sums for the BDD builder";
      return res;
    }
  }
  // 2. codes bottom-up
  sc.code.assign(sc.sums.size(), kCodeBot);
  for (size_t q = sc.lvl[k]; q < sc.lvl[k + 1]; ++q) sc.code[q] = row_holds(sc.sums[q], sense, rhs) ? kCodeTop : kCodeBot;
  if (sc.level_keys.size() < (size_t)k) sc.level_keys.resize(k);
  for (int h = k - 1; h >= 0; --h) {
    const size_t b = sc.lvl[h], e = sc.lvl[h + 1];
    const size_t nb = sc.lvl[h + 1], ne = sc.lvl[h + 2];
    const int64_t* nxt = sc.sums.data() + nb;
    const size_t nn = ne - nb;
    sc.keys.resize(e - b);
    for (size_t q = b; q < e; ++q) {
      const int64_t s = sc.sums[q];
      size_t i0 = std::lower_bound(nxt, nxt + nn, clamp(s, h + 1)) - nxt;
      size_t i1 = std::lower_bound(nxt, nxt + nn, clamp(s + a[h], h + 1)) - nxt;
      const int c0 = sc.code[nb + i0], c1 = sc.code[nb + i1];
      sc.keys[q - b] = (uint64_t(uint32_t(c0 + 2)) << 32) | uint64_t(uint32_t(c1 + 2));
    }
    std::vector<uint64_t>& uniq = sc.level_keys[h];
    uniq.assign(sc.keys.begin(), sc.keys.end());
    std::sort(uniq.begin(), uniq.end());
    uniq.erase(std::unique(uniq.begin(), uniq.end()), uniq.end());
    if (!uniq.empty() && uniq.front() == 0u) uniq.erase(uniq.begin());  // (bottom, bottom)
    for (size_t q = b; q < e; ++q) {
      const uint64_t key = sc.keys[q - b];
      sc.code[q] = key == 0u ? kCodeBot : int(std::lower_bound(uniq.begin(), uniq.end(), key) - uniq.begin());
    }
  }
  if (sc.code[0] == kCodeBot) {
    res.status = DG_EINFEASIBLE;
    res.msg = "row has no feasible assignment";
    return res;
  }
  sc.nodes = 0;
  sc.maxw = 0;
  for (int h = 0; h < k; ++h) {
    bool zero_ok = false, one_ok = false;
    for (uint64_t key : sc.level_keys[h]) {
      zero_ok |= key_lo(key) != kCodeBot;
      one_ok |= key_hi(key) != kCodeBot;
    }
    if (!zero_ok || !one_ok) {
      res.status = DG_EFORCED;
      res.msg = "row fixes one of its variables (presolve it away)";
      return res;
    }
    sc.nodes += (int64_t)sc.level_keys[h].size();
    sc.maxw = std::max<int>(sc.maxw, (int)sc.level_keys[h].size());
  }
  return res;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Shape of a unit row as the unit kernels sweep it, before it has a place in
// the arena.
struct UnitRow {
  UnitShape s{};
  std::vector<uint8_t> type;  // per level
};

inline int unit_z(int t, int u) { return t == kSwap ? std::max(u - 1, 0) : u; }
inline int unit_o(int t, int u) {
  return t == kUp ? u + 1 : (t == kSwap ? u : (t == kDown ? std::max(u - 1, 0) : u - 1));
}

// Tries to read the row sum_h a_h x_h (<= or =) rhs, all a_h = +-1, as a unit
// row (see UnitShape) whose states are the nodes of its canonical BDD
// (level_keys, k levels).  Every arc of the BDD is compared with the shape.
bool unit_candidate(const int8_t* a, int k, bool eq, int64_t rhs, const std::vector<std::vector<uint64_t>>& level_keys,
                    int max_w, UnitRow& out) {
  // sums from which every completion is feasible act like clamp[g] ('<='),
  // those outside the alive range like the bottom
  std::vector<int64_t> pos(k + 1, 0), neg(k + 1, 0);
  for (int h = k - 1; h >= 0; --h) {
    pos[h] = pos[h + 1] + (a[h] > 0);
    neg[h] = neg[h + 1] + (a[h] < 0);
  }
  auto clamp_at = [&](int g) { return eq ? INT64_MIN / 4 : rhs - pos[g]; };
  std::vector<int64_t> l(k + 1), hi(k + 1);
  l[0] = hi[0] = std::max<int64_t>(0, clamp_at(0));
  for (int g = 0; g <= k; ++g) {
    if (g > 0) {
      l[g] = l[g - 1] - (a[g - 1] < 0);
      hi[g] = hi[g - 1] + (a[g - 1] > 0);
    }
    hi[g] = std::max(std::min(hi[g], rhs + neg[g]), clamp_at(g));
    l[g] = std::max(l[g], eq ? rhs - pos[g] : clamp_at(g));
    if (l[g] > hi[g]) return false;
  }
  int64_t smin = l[0];
  for (int g = 0; g < k; ++g) smin = std::min(smin, l[g]);
  std::vector<int64_t> base(k + 1);
  for (int g = 0; g < k; ++g) base[g] = std::max(smin, clamp_at(g));
  base[k] = base[k - 1];
  int64_t W = 1;
  for (int g = 0; g < k; ++g) W = std::max(W, hi[g] - base[g] + 1);
  W = std::max(W, hi[k] - base[k] + 1);
  if (W > max_w) return false;
  UnitShape& s = out.s;
  s.W = 2;
  while (s.W < W) s.W += max_w > kUnitMaxW ? s.W : 2;  // the long rows' windows are powers of two
  s.k = k;
  s.start = (int32_t)(l[0] - base[0]);
  s.accept = 0;
  for (int u = 0; u < s.W; ++u)
    if (eq ? base[k] + u == rhs : base[k] + u <= rhs) s.accept = (int32_t)((uint32_t)s.accept | 1u << u);
  out.type.assign(k, 0);
  for (int h = 0; h < k; ++h) {
    const int64_t shift = base[h + 1] - base[h];
    if (shift < 0 || shift > (a[h] > 0 ? 1 : 0)) return false;
    out.type[h] = (uint8_t)(a[h] > 0 ? (shift == 0 ? kUp : kSwap) : (eq ? kDrop : kDown));
  }
  s.types = 0;
  for (int h = 0; h < std::min(k, kShortK); ++h) s.types |= out.type[h] << (2 * h);
  if (!unit_short(s)) s.types = 0;
  s.rows = -1;
  for (int h = 0, b = 0; h < k; ++h)
    if (h + 1 == k || out.type[h + 1] != out.type[h]) {
      s.rows += (h + 1 - b + 1) / 2;
      b = h + 1;
    }
  // the shape's own feasibility, then every node and arc of the BDD
  std::vector<uint32_t> alive(k + 1);
  alive[k] = (uint32_t)s.accept;
  for (int h = k - 1; h >= 0; --h) {
    alive[h] = 0;
    for (int u = 0; u < s.W; ++u) {
      const int z = unit_z(out.type[h], u), o = unit_o(out.type[h], u);
      if (((alive[h + 1] >> z) & 1) || (o >= 0 && o < s.W && ((alive[h + 1] >> o) & 1))) alive[h] |= 1u << u;
    }
  }
  std::vector<int> at(1, s.start), next;
  if (level_keys[0].size() != 1 || !((alive[0] >> s.start) & 1)) return false;
  for (int h = 0; h < k; ++h) {
    const std::vector<uint64_t>& keys = level_keys[h];
    next.assign(h + 1 < k ? level_keys[h + 1].size() : 0, -1);
    for (size_t r = 0; r < keys.size(); ++r) {
      if (at[r] < 0 || (r > 0 && at[r] >= at[r - 1])) return false;  // ranks descend in u
      for (int beta = 0; beta < 2; ++beta) {
        const int child = beta ? key_hi(keys[r]) : key_lo(keys[r]);
        const int t = beta ? unit_o(out.type[h], at[r]) : unit_z(out.type[h], at[r]);
        const bool live = t >= 0 && t < s.W && ((alive[h + 1] >> t) & 1);
        if ((child != kCodeBot) != live) return false;
        if (!live) continue;
        if (h + 1 == k) {
          if (child != kCodeTop) return false;
        } else {
          if (child < 0 || (next[child] >= 0 && next[child] != t)) return false;
          next[child] = t;
        }
      }
    }
    at.swap(next);
  }
  return true;
}

bool unit_row(const int32_t* a, int k, int sense, int64_t rhs, const std::vector<std::vector<uint64_t>>& level_keys,
              int max_w, UnitRow& out) {
  std::vector<int8_t> sign(k);
  for (int h = 0; h < k; ++h) {
    if (a[h] != 1 && a[h] != -1) return false;
    sign[h] = (int8_t)(sense == 1 ? -a[h] : a[h]);
  }
  if (sense != 2) return unit_candidate(sign.data(), k, false, sense == 1 ? -rhs : rhs, level_keys, max_w, out);
  if (unit_candidate(sign.data(), k, true, rhs, level_keys, max_w, out)) return true;
  for (int h = 0; h < k; ++h) sign[h] = (int8_t)-sign[h];
  return unit_candidate(sign.data(), k, true, -rhs, level_keys, max_w, out);
}

// A row's BDD as the builder keeps it for later rows with the same terms.
struct RowBdd {
  std::vector<std::vector<uint64_t>> level_keys;
  int64_t nodes = 0;
  int maxw = 0;
  int unit = -1;  // index into the building thread's unit shapes
};
// ... up to kRowCache of them per building thread, none larger than this
constexpr size_t kRowCache = 4096;
constexpr int kRowCacheTerms = 512;
constexpr int64_t kRowCacheNodes = 2048;

}  // namespace

dg_status build_plan(const dg_rows* R, const dg_options* opts, Plan& P) {
  if (!R || !R->row_ptr || !R->col || !R->coef || !R->sense || !R->rhs || !R->c)
    return fail(DG_EINVAL, "dg_plan: null row array");
  const int32_t n = R->n;
  const int64_t m = R->m;
  if (n < 0 || m < 0) return fail(DG_EINVAL, "dg_plan: negative sizes");
  if (opts && opts->long_lanes != 0 &&
      (opts->long_lanes < 0 || opts->long_lanes > kWarp || (opts->long_lanes & (opts->long_lanes - 1)) != 0))
    return fail(DG_EINVAL, "dg_plan: long_lanes must be 0 or a power of two up to 32");
  if (R->row_ptr[0] != 0) return fail(DG_EINVAL, "dg_plan: row_ptr[0] must be 0");
  const int64_t nnz = R->row_ptr[m];
  if (nnz > (int64_t)INT32_MAX / 2) return fail(DG_EINVAL, "dg_plan: too many nonzeros");
  for (int64_t j = 0; j < m; ++j) {
    const int64_t b = R->row_ptr[j], e = R->row_ptr[j + 1];
    if (e <= b) return fail(DG_EINVAL, "dg_plan: empty row " + std::to_string(j));
    if (e - b > 4096) return fail(DG_EINVAL, "dg_plan: row longer than 4096 variables");
    if (R->sense[j] < 0 || R->sense[j] > 2) return fail(DG_EINVAL, "dg_plan: sense must be 0, 1 or 2");
    for (int64_t s = b; s < e; ++s) {
      if (R->col[s] < 0 || R->col[s] >= n || (s > b && R->col[s] <= R->col[s - 1]))
        return fail(DG_EINVAL, "dg_plan: columns of row " + std::to_string(j) + " must be ascending ids in [0,n)");
    }
  }
  for (int32_t i = 0; i < n; ++i)
    if (!(R->c[i] == R->c[i]) || R->c[i] == 1.0 / 0.0 || R->c[i] == -1.0 / 0.0)
      return fail(DG_EINVAL, "dg_plan: non-finite cost");
  // instances
  int32_t ni = R->num_inst <= 1 || !R->inst_row_ptr || !R->inst_var_ptr ? 1 : R->num_inst;
  P.inst_row_ptr.resize(ni + 1);
  P.inst_var_ptr.resize(ni + 1);
  if (ni == 1) {
    P.inst_row_ptr = {0, m};
    P.inst_var_ptr = {0, n};
  } else {
    for (int k = 0; k <= ni; ++k) {
      P.inst_row_ptr[k] = R->inst_row_ptr[k];
      P.inst_var_ptr[k] = R->inst_var_ptr[k];
    }
    if (P.inst_row_ptr[0] != 0 || P.inst_row_ptr[ni] != m || P.inst_var_ptr[0] != 0 || P.inst_var_ptr[ni] != n)
      return fail(DG_EINVAL, "dg_plan: instance pointers must span all rows and variables");
    for (int k = 0; k < ni; ++k) {
      if (P.inst_row_ptr[k + 1] < P.inst_row_ptr[k] || P.inst_var_ptr[k + 1] < P.inst_var_ptr[k])
        return fail(DG_EINVAL, "dg_plan: instance pointers must be non-decreasing");
      for (int64_t j = P.inst_row_ptr[k]; j < P.inst_row_ptr[k + 1]; ++j)
        for (int64_t s = R->row_ptr[j]; s < R->row_ptr[j + 1]; ++s)
          if (R->col[s] < P.inst_var_ptr[k] || R->col[s] >= P.inst_var_ptr[k + 1])
            return fail(DG_EINVAL, "dg_plan: row uses a variable of another instance");
    }
  }

  // ---- 1. BDDs, in parallel over contiguous row ranges --------------------
  int nthreads = opts && opts->num_threads > 0 ? opts->num_threads : (int)std::thread::hardware_concurrency();
  nthreads = std::max(1, std::min<int>(nthreads, (int)std::max<int64_t>(1, std::min<int64_t>(m / 64, nnz / 16384))));
  struct Part {
    std::vector<uint8_t> width;
    std::vector<int8_t> lo, hi;
    std::vector<int32_t> nodes_of_row;
    std::vector<int32_t> unit_of_row;  // index into `units`, -1 for other rows
    std::vector<UnitRow> units;        // distinct unit shapes, by first row
    // rows whose BDD exceeds the tile limits: row, level widths, child ranks
    std::vector<int64_t> long_rows;
    std::vector<int32_t> lwidth, llo, lhi;
    RowResult err;
    int64_t err_row = -1;
  };
  std::vector<Part> parts(nthreads);
  std::vector<int64_t> cut(nthreads + 1);
  for (int t = 0; t <= nthreads; ++t) cut[t] = m * t / nthreads;
  auto worker = [&](int t) {
    RowScratch sc;
    Part& pt = parts[t];
    pt.nodes_of_row.reserve(cut[t + 1] - cut[t]);
    pt.unit_of_row.reserve(cut[t + 1] - cut[t]);
    // most rows of an instance repeat a few (coefficients, sense, rhs): their
    // BDD is built once per thread
    std::unordered_map<std::string, RowBdd> cache;
    std::unordered_map<std::string, int> unit_index;
    std::string key;
    RowBdd built;
    for (int64_t j = cut[t]; j < cut[t + 1]; ++j) {
      const int64_t b = R->row_ptr[j];
      const int k = (int)(R->row_ptr[j + 1] - b);
      const RowBdd* bdd = nullptr;
      if (k <= kRowCacheTerms) {
        key.assign((const char*)(R->coef + b), (size_t)k * 4);
        key.append((const char*)&R->rhs[j], 4);
        key.push_back((char)R->sense[j]);
        auto it = cache.find(key);
        if (it != cache.end()) bdd = &it->second;
      }
      if (!bdd) {
        RowResult r = build_row(R->coef + b, k, R->sense[j], R->rhs[j], sc);
        if (r.status != 0) {
          pt.err = r;
          pt.err_row = j;
          return;
        }
        built.level_keys.assign(sc.level_keys.begin(), sc.level_keys.begin() + k);
        built.nodes = sc.nodes;
        built.maxw = sc.maxw;
        built.unit = -1;
        UnitRow u;
        const bool tile = sc.nodes <= kMaxNodesPerBdd && sc.maxw <= kMaxWidth;
        const int max_w = tile ? kUnitMaxW : kLongUnitMaxW;
        if (sc.maxw <= max_w && (tile || k <= kLongUnitMaxK) &&
            unit_row(R->coef + b, k, R->sense[j], R->rhs[j], built.level_keys, max_w, u)) {
          std::string uk((const char*)&u.s, sizeof(UnitShape));
          uk.append((const char*)u.type.data(), u.type.size());
          auto at = unit_index.emplace(uk, (int)pt.units.size());
          if (at.second) pt.units.push_back(u);
          built.unit = at.first->second;
        }
        if (k <= kRowCacheTerms && built.nodes <= kRowCacheNodes && cache.size() < kRowCache)
          bdd = &cache.emplace(key, std::move(built)).first->second;
        else
          bdd = &built;
      }
      pt.unit_of_row.push_back(bdd->unit);
      if (bdd->nodes <= kMaxNodesPerBdd && bdd->maxw <= kMaxWidth) {
        for (int h = 0; h < k; ++h) {
          pt.width.push_back((uint8_t)bdd->level_keys[h].size());
          for (uint64_t key : bdd->level_keys[h]) {
            pt.lo.push_back((int8_t)key_lo(key));
            pt.hi.push_back((int8_t)key_hi(key));
          }
        }
        pt.nodes_of_row.push_back((int32_t)bdd->nodes);
      } else {
        pt.width.insert(pt.width.end(), (size_t)k, (uint8_t)0);
        pt.nodes_of_row.push_back(0);
        pt.long_rows.push_back(j);
        for (int h = 0; h < k; ++h) {
          pt.lwidth.push_back((int32_t)bdd->level_keys[h].size());
          for (uint64_t key : bdd->level_keys[h]) {
            pt.llo.push_back(key_lo(key));
            pt.lhi.push_back(key_hi(key));
          }
        }
      }
    }
  };
  if (nthreads == 1) {
    worker(0);
  } else {
    std::vector<std::thread> th;
    for (int t = 0; t < nthreads; ++t) th.emplace_back(worker, t);
    for (auto& x : th) x.join();
  }
  for (int t = 0; t < nthreads; ++t)
    if (parts[t].err.status != 0)
      return fail((dg_status)parts[t].err.status, "dg_plan: row " + std::to_string(parts[t].err_row) + ": " +
                                                      parts[t].err.msg);
  std::vector<uint8_t> width;
  width.reserve(nnz);
  P.node_ptr.assign(m + 1, 0);
  std::vector<int64_t> long_rows;
  std::vector<int32_t> long_width;  // level widths of the long BDDs, in row order
  std::vector<UnitRow> units;       // distinct unit shapes, by first row
  std::vector<int32_t> unit_of_row(m, -1);
  {
    std::unordered_map<std::string, int> unit_index;
    int64_t j = 0;
    for (int t = 0; t < nthreads; ++t) {
      width.insert(width.end(), parts[t].width.begin(), parts[t].width.end());
      P.lo8.insert(P.lo8.end(), parts[t].lo.begin(), parts[t].lo.end());
      P.hi8.insert(P.hi8.end(), parts[t].hi.begin(), parts[t].hi.end());
      std::vector<int> global;
      for (const UnitRow& u : parts[t].units) {
        std::string uk((const char*)&u.s, sizeof(UnitShape));
        uk.append((const char*)u.type.data(), u.type.size());
        auto at = unit_index.emplace(uk, (int)units.size());
        if (at.second) units.push_back(u);
        global.push_back(at.first->second);
      }
      for (size_t x = 0; x < parts[t].nodes_of_row.size(); ++x) {
        const int u = parts[t].unit_of_row[x];
        if (u >= 0) unit_of_row[j] = global[u];
        P.node_ptr[j + 1] = P.node_ptr[j] + parts[t].nodes_of_row[x];
        ++j;
      }
      long_rows.insert(long_rows.end(), parts[t].long_rows.begin(), parts[t].long_rows.end());
      long_width.insert(long_width.end(), parts[t].lwidth.begin(), parts[t].lwidth.end());
      P.long_lo.insert(P.long_lo.end(), parts[t].llo.begin(), parts[t].llo.end());
      P.long_hi.insert(P.long_hi.end(), parts[t].lhi.begin(), parts[t].lhi.end());
      std::vector<uint8_t>().swap(parts[t].width);
      std::vector<int8_t>().swap(parts[t].lo);
      std::vector<int8_t>().swap(parts[t].hi);
      std::vector<int32_t>().swap(parts[t].llo);
      std::vector<int32_t>().swap(parts[t].lhi);
    }
  }
  P.row_ptr.assign(R->row_ptr, R->row_ptr + m + 1);
  P.long_of_row.assign(m, -1);
  for (size_t b = 0; b < long_rows.size(); ++b) P.long_of_row[long_rows[b]] = (int32_t)b;
  const int64_t num_long_nodes = (int64_t)P.long_lo.size();
  const int64_t num_nodes = P.node_ptr[m] + num_long_nodes;

  // ---- 2. tiles: 32 BDDs per tile, one per lane ---------------------------
  // Rows are cut into chunks of consecutive rows (so that a tile's variables,
  // and the S values its lanes gather, stay close together).  The unit rows of
  // one shape fill tiles of their own, in row order whatever the chunk; theirs
  // is kUnitChunk rows at least, since every chunk leaves a tile per shape partly
  // filled.  The other rows are sorted by hop count and node count inside a
  // chunk, longest first, and every 32 consecutive ones form a tile.  Inside a tile everything is interleaved by
  // lane: slot (h, b) is slot_base + 32 h + b and node number n of lane b is
  // element 32 n + b of the per-tile arrays.  Node numbers 0 and 1 stand for
  // the top and bottom terminals, the BDD's own nodes are numbered 2, 3, ...
  // level by level; child codes are node numbers (8 bits).
  // Rows of the long BDDs take no tile (they are laid out after the tiles).
  constexpr int64_t kUnitChunk = 16384;
  const int64_t kChunkRows = opts && opts->chunk_rows > 0 ? opts->chunk_rows : kUnitChunk;
  struct TileSrc {
    int64_t first;  // its rows: order[first .. first + count)
    int count, unit;
  };
  std::vector<int64_t> order;
  std::vector<TileSrc> src;
  order.reserve(m - (int64_t)long_rows.size());
  {
    // a shape's last tile is rarely full.  It becomes a unit tile of its own
    // when at least half its lanes are in use, or while a chunk has few such
    // tiles (an empty lane costs memory, a mixed tile several times a unit
    // tile's time); the rows of the others join the mixed tiles
    constexpr int kHalf = kWarp / 2, kFewPartial = 64;
    std::vector<std::pair<int32_t, int64_t>> by_shape;
    std::vector<int64_t> mixed;
    std::vector<TileSrc> part;
    const int64_t step = std::max(kChunkRows, kUnitChunk);
    for (int64_t c0 = 0; c0 < m; c0 += step) {
      const int64_t c1 = std::min(m, c0 + step);
      by_shape.clear();
      part.clear();
      for (int64_t j = c0; j < c1; ++j) {
        if (P.long_of_row[j] >= 0) continue;
        if (unit_of_row[j] >= 0)
          by_shape.emplace_back(unit_of_row[j], j);
        else
          mixed.push_back(j);
      }
      std::sort(by_shape.begin(), by_shape.end());
      size_t full = 0;
      for (size_t x = 0; x < by_shape.size();) {
        size_t e = x;
        while (e < by_shape.size() && e - x < (size_t)kWarp && by_shape[e].first == by_shape[x].first) ++e;
        if (e - x == (size_t)kWarp) {
          src.push_back({(int64_t)order.size(), kWarp, by_shape[x].first});
          for (size_t y = x; y < e; ++y) order.push_back(by_shape[y].second);
          ++full;
        } else {
          part.push_back({(int64_t)x, (int)(e - x), by_shape[x].first});
        }
        x = e;
      }
      std::stable_sort(part.begin(), part.end(), [](const TileSrc& x, const TileSrc& y) { return x.count > y.count; });
      for (size_t i = 0; i < part.size(); ++i) {
        const TileSrc& t = part[i];
        const bool own = t.count >= kHalf || i < std::max<size_t>(kFewPartial, full / 8);
        if (own) src.push_back({(int64_t)order.size(), t.count, t.unit});
        for (int64_t y = t.first; y < t.first + t.count; ++y)
          (own ? order : mixed).push_back(by_shape[y].second);
      }
    }
    std::sort(mixed.begin(), mixed.end(), [&](int64_t x, int64_t y) {
      if (x / kChunkRows != y / kChunkRows) return x < y;
      const int64_t kx = R->row_ptr[x + 1] - R->row_ptr[x], ky = R->row_ptr[y + 1] - R->row_ptr[y];
      if (kx != ky) return kx > ky;
      const int64_t nx = P.node_ptr[x + 1] - P.node_ptr[x], ny = P.node_ptr[y + 1] - P.node_ptr[y];
      return nx != ny ? nx > ny : x < y;
    });
    for (size_t x = 0; x < mixed.size(); x += kWarp) {
      const size_t e = std::min(mixed.size(), x + kWarp);
      src.push_back({(int64_t)order.size(), (int)(e - x), -1});
      order.insert(order.end(), mixed.begin() + x, mixed.begin() + e);
    }
  }
  int max_hops = 0, max_width = 0;
  for (int64_t j = 0; j < m; ++j) {
    int k = (int)(R->row_ptr[j + 1] - R->row_ptr[j]);
    max_hops = std::max(max_hops, k);
    P.hop_histogram[std::min(k, 63)]++;
  }
  for (uint8_t w : width) max_width = std::max<int>(max_width, w);
  for (int32_t w : long_width) max_width = std::max<int>(max_width, w);

  const int T = (int)src.size();
  if (opts && opts->host_mb_limit > 0) {
    // host bytes of the arena image about to be built: child codes, slot
    // arrays (descriptor, variable, row, CSR position), variable CSR and ELL
    const double est = 2.0 * (double)num_nodes * 1.1 + 18.0 * (double)nnz * 1.1 + 8.0 * (double)nnz +
                       (16.0 + 4.0 * kEll) * (double)n + 40.0 * (double)T;
    if (est > (double)opts->host_mb_limit * 1048576.0)
      return fail(DG_ENOMEM, "dg_plan: the arena image needs about " + std::to_string((long long)(est / 1048576.0)) +
                                 " MiB of host memory, more than host_mb_limit");
  }
  // tiles are laid out by shared-memory footprint, largest first (the unit
  // tiles, then the others), so that tiles of one launch group are contiguous
  // and the longest tiles start first
  std::vector<int> tile_nh(T, 0), tile_nmax(T, 2), tile_maxw(T, 1), tile_order(T);
  for (int t = 0; t < T; ++t) {
    for (int64_t q = src[t].first; q < src[t].first + src[t].count; ++q) {
      const int64_t j = order[q];
      tile_nh[t] = std::max<int>(tile_nh[t], (int)(R->row_ptr[j + 1] - R->row_ptr[j]));
      tile_nmax[t] = std::max<int>(tile_nmax[t], 2 + (int)(P.node_ptr[j + 1] - P.node_ptr[j]));
      for (int64_t c = R->row_ptr[j]; c < R->row_ptr[j + 1]; ++c) tile_maxw[t] = std::max<int>(tile_maxw[t], width[c]);
    }
    tile_order[t] = t;
  }
  auto tile_smem = [&](int t) {
    return src[t].unit >= 0 ? unit_smem_bytes(units[src[t].unit].s, 1)
                            : sweep_smem_bytes(tile_nmax[t], tile_nh[t], 1, ring_size(tile_maxw[t]));
  };
  int nunit = 0, nshort = 0;
  size_t largest = 1;  // footprint
  for (int t = 0; t < T; ++t) {
    nunit += src[t].unit >= 0;
    nshort += src[t].unit >= 0 && unit_short(units[src[t].unit].s);
    largest = std::max(largest, tile_smem(t));
  }
  // An arena of unit tiles alone is one launch (then chained, see Plan::chained)
  // while its tiles, at the largest one's footprint, fill the chip at most
  // kOneLaunchFills times and that footprint leaves at least seven warps per SM.
  // us per iteration (plain; per slot; recorded and reversed), one launch /
  // several forked: tracking with 50 frames of 400 detections 17; 18; 53 / 29;
  // 29; 75, 25 frames of 2,000, 2.8 fills 33; 34; 90 / 38; 40; 98, 50 frames, 5.2
  // fills 49; 54; 152 / 51; 59; 153, 80 frames, 10 fills 70; 85; 253 / 70; 77; 224.
  constexpr size_t kSmSmem = 224 * 1024, kOneLaunchFills = 6, kOneLaunchSmem = 32 * 1024;
  const bool one_launch = nunit == T && long_rows.empty() && largest <= kOneLaunchSmem &&
                          (size_t)T <= kOneLaunchFills * kSms * std::min<size_t>(64, kSmSmem / largest);
  // The kernels for short unit tiles take them where they are most of the unit
  // tiles.  As one more launch group they cost a few microseconds a sweep (the
  // launch, or the fork and join of a stream), so only where they are all, or
  // next to many others, and where that is not one launch more.  us an iteration
  // without and with them: batch of 64 mixed instances, replayed from a graph,
  // 159 / 144; of 8, 12,300 tiles, one launch without, 37 / 43; of 4 19 / 33;
  // matching 16 / 20.
  constexpr int kShortTiles = 8192;
  const bool short_kernels = nshort == nunit || (2 * nshort >= nunit && nunit >= kShortTiles && !one_launch);
  // (kind 0: unit tiles, 1: short unit tiles, 2: mixed tiles)
  auto tile_kind = [&](int t) {
    return src[t].unit < 0 ? 2 : (short_kernels && unit_short(units[src[t].unit].s) ? 1 : 0);
  };
  std::stable_sort(tile_order.begin(), tile_order.end(), [&](int x, int y) {
    const int kx = tile_kind(x), ky = tile_kind(y);
    return kx != ky ? kx < ky : tile_smem(x) > tile_smem(y);
  });
  // the shapes in use, in tile order
  std::vector<int> shape_slot(units.size(), -1);
  P.unit_shapes.clear();
  P.unit_runs.clear();
  for (int t : tile_order) {
    const int u = src[t].unit;
    if (u < 0 || shape_slot[u] >= 0) continue;
    shape_slot[u] = (int)P.unit_shapes.size();
    UnitShape s = units[u].s;
    s.run_base = (int32_t)P.unit_runs.size();
    for (int h = 0; h < s.k; ++h)
      if (h + 1 == s.k || units[u].type[h + 1] != units[u].type[h])
        P.unit_runs.push_back((uint16_t)((h + 1) << 2 | units[u].type[h]));
    s.nruns = (int32_t)P.unit_runs.size() - s.run_base;
    P.unit_shapes.push_back(s);
  }
  P.tiles.resize(T);
  P.slot_to_csr.clear();
  std::vector<int64_t> slot_of_csr(nnz, -1);
  int64_t node_base = 0, slot_base = 0;
  size_t smem_max = 0, smem_adj_max = 0;
  for (int t = 0; t < T; ++t) {
    const int ts = tile_order[t];
    const int64_t q0 = src[ts].first;
    const int nb = src[ts].count;
    const int nh = tile_nh[ts], nmax = tile_nmax[ts];
    const int64_t tslots = (int64_t)nh * kWarp;
    Tile& tile = P.tiles[t];
    tile.unit = src[ts].unit >= 0 ? 1 + shape_slot[src[ts].unit] : 0;
    tile.node_base = (int32_t)node_base;
    tile.slot_base = (int32_t)slot_base;
    tile.nmax = nmax;
    tile.nhops = nh;
    tile.nbdd = nb;
    int maxw = 1;
    P.desc.resize(slot_base + tslots, 0);
    P.slot_var.resize(slot_base + tslots, -1);
    P.slot_row.resize(slot_base + tslots, -1);
    P.slot_to_csr.resize(slot_base + tslots, -1);
    P.lohi8.resize(node_base + (int64_t)(nmax - 2) * kWarp, 0x0101u);
    for (int bb = 0; bb < nb; ++bb) {
      const int64_t j = order[q0 + bb];
      const int k = (int)(R->row_ptr[j + 1] - R->row_ptr[j]);
      const int64_t nbj = P.node_ptr[j];
      int first = 2;
      for (int h = 0; h < k; ++h) {
        const int64_t csr = R->row_ptr[j] + h;
        const int w = width[csr];
        maxw = std::max(maxw, w);
        const int64_t sl = slot_base + (int64_t)h * kWarp + bb;
        P.desc[sl] = (uint16_t)(first | (w << 8));
        P.slot_var[sl] = R->col[csr];
        P.slot_row[sl] = (int32_t)j;
        P.slot_to_csr[sl] = csr;
        slot_of_csr[csr] = sl;
        const int first_next = first + w;
        for (int r = 0; r < w; ++r) {
          auto code = [&](int8_t cc) -> uint32_t {
            return cc == kCodeBot ? kBotCode : (cc == kCodeTop ? kTopCode : (uint32_t)(first_next + cc));
          };
          const int64_t nidx = nbj + (first - 2) + r;
          P.lohi8[node_base + (int64_t)(first - 2 + r) * kWarp + bb] =
              (uint16_t)(code(P.lo8[nidx]) | (code(P.hi8[nidx]) << 8));
        }
        first = first_next;
      }
    }
    tile.maxw = maxw;
    tile.ring = ring_size(maxw);
    smem_max = std::max(smem_max, sweep_smem_bytes(nmax, nh, 1, tile.ring));
    smem_adj_max = std::max(smem_adj_max, adjoint_smem_bytes(nmax, nh));
    P.max_tile_rows = std::max(P.max_tile_rows, nmax);
    P.max_tile_slots = std::max<int32_t>(P.max_tile_slots, (int32_t)tslots);
    P.max_tile_hops = std::max(P.max_tile_hops, nh);
    node_base += (int64_t)(nmax - 2) * kWarp;
    slot_base += tslots;
    if (tile.unit) {
      P.unit_slots = (int32_t)slot_base;
      P.unit_nodes = (int32_t)node_base;
    }
  }
  // launch groups: consecutive tiles whose footprints stay within 1/kGroupRatio
  // of the group's largest one
  {
    const double kGroupRatio =
        opts && opts->group_ratio_pct > 0 && opts->group_ratio_pct <= 100 ? opts->group_ratio_pct / 100.0 : 0.85;
    // ... or any smaller one while the group's tiles do not fill the chip (its
    // smaller tiles then cost it no occupancy and save a launch)
    // ... but no tile that would keep the group's recording sweeps from fitting a
    // CTA: these take the largest footprint and the largest records together
    constexpr size_t kCtaSmem = 227 * 1024;
    int32_t t0 = 0;
    size_t gmax = 0, rec_max = 0, meta_max = 0;
    auto group_smem = [&](int t) {
      const Tile& tl = P.tiles[t];
      return tl.unit ? unit_smem_bytes(P.unit_shapes[tl.unit - 1], 1)
                     : sweep_smem_bytes(tl.nmax, tl.nhops, 1, tl.ring);
    };
    auto group_kind = [&](int t) {
      const Tile& tl = P.tiles[t];
      return !tl.unit ? 2 : (short_kernels && unit_short(P.unit_shapes[tl.unit - 1]) ? 1 : 0);
    };
    for (int t = 0; t <= T; ++t) {
      const size_t r = t < T ? group_smem(t) : 0;
      const bool full = gmax > 0 && (size_t)(t - t0) >= kSms * std::min<size_t>(64, kSmSmem / gmax);
      // (short unit tiles need no shared memory: one group whatever their size)
      const int kind = t < T ? group_kind(t) : 3, kind0 = t > t0 ? group_kind(t0) : kind;
      size_t rec = 0, meta = 0;
      if (kind == 2) {
        const Tile& tl = P.tiles[t];
        rec = std::max(r, sweep_smem_bytes_bwd(tl.nmax, tl.nhops, 1));
        meta = (size_t)(tl.nmax - 2) * kWarp * 2;
      }
      const bool cut = kind != kind0 || (kind != 1 && full && !one_launch && (double)r < kGroupRatio * (double)gmax) ||
                       (std::max(rec, rec_max) + std::max(meta, meta_max) > kCtaSmem && rec + meta <= kCtaSmem);
      if (t == T || (t > t0 && cut)) {
        if (t > t0) {
          LaunchGroup g{};
          g.tile0 = t0;
          g.tile1 = t;
          P.groups.push_back(g);
        }
        t0 = t;
        gmax = rec_max = meta_max = 0;
      }
      gmax = std::max(gmax, r);
      rec_max = std::max(rec_max, rec);
      meta_max = std::max(meta_max, meta);
    }
    for (LaunchGroup& g : P.groups)
      for (int t = g.tile0; t < g.tile1; ++t) {
        const Tile& tl = P.tiles[t];
        g.region_bytes = std::max<int32_t>(g.region_bytes, (int32_t)sweep_smem_bytes(tl.nmax, tl.nhops, 1, tl.ring));
        g.region_bytes0 = std::max<int32_t>(g.region_bytes0, (int32_t)sweep_smem_bytes(tl.nmax, tl.nhops, 0, tl.ring));
        if (tl.unit) {
          const UnitShape& s = P.unit_shapes[tl.unit - 1];
          g.unit_w = std::max(g.unit_w, s.W);
          g.unit_short = short_kernels && unit_short(s);  // as all of the group
          g.unit_bytes0 = std::max<int32_t>(g.unit_bytes0, (int32_t)unit_smem_bytes(s, 0));
          g.unit_bytes1 = std::max<int32_t>(g.unit_bytes1, (int32_t)unit_smem_bytes(s, 1));
        }
        g.region_bwd1 = std::max<int32_t>(g.region_bwd1, (int32_t)sweep_smem_bytes_bwd(P.tiles[t].nmax, P.tiles[t].nhops, 1));
        g.region_bwd0 = std::max<int32_t>(g.region_bwd0, (int32_t)sweep_smem_bytes_bwd(P.tiles[t].nmax, P.tiles[t].nhops, 0));
        g.meta_bytes = std::max<int32_t>(g.meta_bytes, (P.tiles[t].nmax - 2) * kWarp * 2);
        smem_max = std::max<size_t>(smem_max, (size_t)std::max(g.region_bwd1, g.unit_bytes1));
      }
    // work estimate per group, then longest-processing-time assignment of the
    // groups to the kStreams streams that run one sweep's launches concurrently
    for (LaunchGroup& g : P.groups)
      for (int t = g.tile0; t < g.tile1; ++t) {
        const Tile& tl = P.tiles[t];
        g.work += tl.unit ? (int64_t)tl.nhops * (14 * P.unit_shapes[tl.unit - 1].W + 40)
                          : (int64_t)kWarp * tl.nmax * tl.nhops;
      }
    // the long BDDs are one more launch (index -1 here): a warp walks each
    // level in turn, estimated like a tile level of 16 nodes per level
    int64_t long_work = 0;
    for (size_t b = 0; b < long_rows.size(); ++b)
      long_work += (int64_t)kWarp * 16 * (R->row_ptr[long_rows[b] + 1] - R->row_ptr[long_rows[b]]);
    auto work_of = [&](int x) { return x < 0 ? long_work : P.groups[x].work; };
    std::vector<int> idx(P.groups.size());
    std::iota(idx.begin(), idx.end(), 0);
    if (!long_rows.empty()) idx.push_back(-1);
    std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return work_of(x) > work_of(y); });
    std::vector<int64_t> load(kStreams, 0);
    for (int gi : idx) {
      int best = 0;
      for (int k = 1; k < kStreams; ++k)
        if (load[k] < load[best]) best = k;
      if (gi < 0)
        P.long_stream = best;
      else
        P.groups[gi].stream = best;
      load[best] += work_of(gi);
    }
  }
  for (const LaunchGroup& g : P.groups) {
    AdjGroup a{g.tile0, g.tile1, 0, g.stream, g.unit_w};
    for (int t = g.tile0; t < g.tile1; ++t)
      a.region = std::max<int32_t>(
          a.region, (int32_t)(g.unit_w ? unit_adjoint_bytes(P.tiles[t].nhops)
                                       : adjoint_smem_bytes(P.tiles[t].nmax, P.tiles[t].nhops)));
    P.adj_groups.push_back(a);
  }
  // ---- 2b. long BDDs: levels as consecutive slots after the tiles (each
  // BDD's range padded to a multiple of 32), nodes numbered 2, 3, ... level
  // by level with 32-bit children (0 top, 1 bottom), and per node its
  // in-arcs in (parent, beta) order
  P.long_slot_base = (int32_t)slot_base;
  {
    int64_t lslot = slot_base, code_base = 0, lvl_base = 0, cost_base = 0, wpos = 0, rpos = 0;
    P.longs.resize(long_rows.size());
    P.long_rank_ptr.assign(long_rows.size() + 1, 0);
    P.long_code.resize(num_long_nodes);
    P.long_in_ptr.assign(num_long_nodes + 1, 0);
    std::vector<int32_t> first;
    for (size_t b = 0; b < long_rows.size(); ++b) {
      const int64_t j = long_rows[b];
      const int k = (int)(R->row_ptr[j + 1] - R->row_ptr[j]);
      LongBdd& L = P.longs[b];
      L.slot_base = (int32_t)lslot;
      L.k = k;
      L.code_base = (int32_t)code_base;
      L.lvl_base = (int32_t)lvl_base;
      L.cost_base = (int32_t)cost_base;
      L.row = (int32_t)j;
      L.maxw = 0;
      first.assign(k + 1, 2);
      for (int h = 0; h < k; ++h) {
        const int w = long_width[wpos + h];
        first[h + 1] = first[h] + w;
        L.maxw = std::max(L.maxw, w);
      }
      L.nn = first[k] - 2;
      P.long_lvl.insert(P.long_lvl.end(), first.begin(), first.end());
      const int64_t tslots = ((int64_t)k + kWarp - 1) / kWarp * kWarp;
      P.desc.resize(lslot + tslots, 0);
      P.slot_var.resize(lslot + tslots, -1);
      P.slot_row.resize(lslot + tslots, -1);
      P.slot_to_csr.resize(lslot + tslots, -1);
      for (int h = 0; h < k; ++h) {
        const int64_t csr = R->row_ptr[j] + h, sl = lslot + h;
        P.slot_var[sl] = R->col[csr];
        P.slot_row[sl] = (int32_t)j;
        P.slot_to_csr[sl] = csr;
        slot_of_csr[csr] = sl;
      }
      // children as node numbers; in-degree counts
      P.long_rank_ptr[b] = rpos;
      for (int h = 0; h < k; ++h)
        for (int r = 0; r < long_width[wpos + h]; ++r) {
          auto num = [&](int32_t rank) -> int32_t {
            return rank == kCodeBot ? (int32_t)kBotCode : (rank == kCodeTop ? (int32_t)kTopCode : first[h + 1] + rank);
          };
          const int32_t lo = num(P.long_lo[rpos]), hi = num(P.long_hi[rpos]);
          int2& cc = P.long_code[code_base + (first[h] - 2) + r];
          cc.x = lo;
          cc.y = hi;
          if (lo >= 2) P.long_in_ptr[code_base + (lo - 2) + 1]++;
          if (hi >= 2) P.long_in_ptr[code_base + (hi - 2) + 1]++;
          ++rpos;
        }
      wpos += k;
      lslot += tslots;
      code_base += L.nn;
      lvl_base += k + 1;
      cost_base += L.nn + 2;
    }
    P.long_rank_ptr[long_rows.size()] = rpos;
    for (int64_t g = 0; g < num_long_nodes; ++g) P.long_in_ptr[g + 1] += P.long_in_ptr[g];
    P.long_in.assign(P.long_in_ptr[num_long_nodes], 0);
    std::vector<int32_t> fill(P.long_in_ptr.begin(), P.long_in_ptr.end() - 1);
    for (const LongBdd& L : P.longs)  // parents ascending, the 0-arc first
      for (int n = 2; n < L.nn + 2; ++n) {
        const int2 c = P.long_code[L.code_base + n - 2];
        if (c.x >= 2) P.long_in[fill[L.code_base + c.x - 2]++] = n << 1;
        if (c.y >= 2) P.long_in[fill[L.code_base + c.y - 2]++] = (n << 1) | 1;
      }
    slot_base = lslot;
    if (cost_base >= (int64_t)INT32_MAX || P.long_in_ptr[num_long_nodes] >= (int64_t)INT32_MAX)
      return fail(DG_EINVAL, "dg_plan: long BDDs exceed 2^31 nodes or arcs");
    P.long_cost_size = (int32_t)cost_base;
    // the plain sweeps pack the narrow long BDDs several to a warp: list them
    // first, longest first (a warp's BDDs then take about as many levels)
    P.long_order.clear();
    for (size_t b = 0; b < P.longs.size(); ++b)
      if (P.longs[b].maxw <= kWarp) P.long_order.push_back((int32_t)b);
    // ... the unit ones by kind before the others
    std::unordered_map<std::string, int> kind_index;
    std::vector<int> kind(P.longs.size(), INT32_MAX);
    for (int32_t b : P.long_order) {
      const int u = unit_of_row[P.longs[b].row];
      if (u < 0) continue;
      const UnitRow& U = units[u];
      const bool one = std::count(U.type.begin(), U.type.end(), U.type[0]) == (std::ptrdiff_t)U.type.size();
      std::string uk((const char*)&U.s.W, 4);
      uk.append((const char*)&U.s.start, 4);
      uk.append((const char*)&U.s.accept, 4);
      uk.append((const char*)U.type.data(), one ? 1 : U.type.size());
      kind[b] = kind_index.emplace(uk, (int)kind_index.size()).first->second;
    }
    std::stable_sort(P.long_order.begin(), P.long_order.end(), [&](int32_t x, int32_t y) {
      return kind[x] != kind[y] ? kind[x] < kind[y] : P.longs[x].k > P.longs[y].k;
    });
    P.num_long_unit = 0;
    for (int32_t b : P.long_order) P.num_long_unit += kind[b] != INT32_MAX;
    P.long_items.clear();
    for (int32_t i = 0; i < P.num_long_unit;) {
      const int k0 = kind[P.long_order[i]];
      int32_t e = i;
      while (e < P.num_long_unit && kind[P.long_order[e]] == k0) ++e;
      const UnitRow& U = units[unit_of_row[P.longs[P.long_order[i]].row]];
      const int G = U.s.W, kmax = P.longs[P.long_order[i]].k;
      // BDDs per warp: as many as lanes allow while that leaves at least four
      // warps per SM (a warp's levels are a chain of dependent steps, which
      // other warps hide), and as fit shared memory
      // (or as many as dg_options::long_lanes asks for)
      const int lanes = opts ? opts->long_lanes : 0;
      int nseg = std::min(G <= kUnitMaxW ? kWarp : kWarp / G, lanes > 0 ? kWarp / lanes : kWarp);
      while (nseg > 1 && ((lanes == 0 && (int64_t)(e - i) < 4LL * kSms * nseg) ||
                          long_unit_bytes(nseg, G, kmax, 1) > 64 * 1024 || long_unit_adjoint_bytes(nseg, kmax) > 64 * 1024))
        nseg /= 2;
      const int32_t run_base = (int32_t)P.unit_runs.size();
      for (int h = 0; h < U.s.k; ++h)
        if (h + 1 == U.s.k || U.type[h + 1] != U.type[h]) P.unit_runs.push_back((uint16_t)((h + 1) << 2 | U.type[h]));
      for (int32_t x = i; x < e; x += nseg) {
        LongItem it{};
        it.first = x;
        it.nseg = std::min(nseg, e - x);
        it.G = G;
        it.kmax = P.longs[P.long_order[x]].k;
        it.start = U.s.start;
        it.accept = (uint32_t)U.s.accept;
        it.run_base = run_base;
        it.nruns = (int32_t)P.unit_runs.size() - run_base;
        P.long_items.push_back(it);
        for (int mode = 0; mode < 2; ++mode)
          P.long_unit_smem[mode] = std::max<int32_t>(P.long_unit_smem[mode], (int32_t)long_unit_bytes(it.nseg, G, it.kmax, mode));
        P.long_unit_adj_smem = std::max<int32_t>(P.long_unit_adj_smem, (int32_t)long_unit_adjoint_bytes(it.nseg, it.kmax));
      }
      i = e;
    }
    // the longest items first
    std::stable_sort(P.long_items.begin(), P.long_items.end(),
                     [](const LongItem& x, const LongItem& y) { return x.kmax > y.kmax; });
    // Plain sweeps of the unit ones.  Their kernels walk every level twice, with
    // the path costs in shared memory, which leaves few warps to an SM when the
    // rows are long and wide; the general kernel takes the costs of the sweep
    // before and needs none.  A sweep's time: levels times a step over the warps
    // an SM holds, against the larger of one row's chain and the SM's rate (ns a
    // level).  us per iteration, unit / general: 13 states, 700 variables, 3,500
    // rows 995 / 1112, 5,000 rows 1478 / 1187; 31 states, 1,000 variables, 1,200
    // rows 1156 / 1472, 2,000 rows 2022 / 1584; 6 states, 1,300 variables, 6,000
    // rows 1941 / 2028; 2 states, 1,300 variables, 20,000 rows 2310 / 4797.
    {
      const double warps = std::min(32, 227 * 1024 / (std::max(P.long_unit_smem[0], 1) + 1024));
      double unit = 0, rate = 0, chain = 0;
      for (const LongItem& it : P.long_items) {
        unit += it.kmax * (it.G <= kUnitMaxW ? 75.0 : (it.G == 16 ? 130.0 : 77.0)) / (warps * kSms);
        rate += (double)it.nseg * it.kmax * (it.G <= kUnitMaxW ? 15.0 : (it.G == 16 ? 24.0 : 45.0)) / kSms;
        chain = std::max(chain, 800.0 * it.kmax);
      }
      P.long_plain = unit > std::max(rate, chain) ? 0 : P.num_long_unit;
    }
    P.chained = P.long_plain == (int32_t)P.longs.size() &&
                (T == 0 || (nunit == T && P.longs.empty() && P.groups.size() == 1));
    P.num_long_narrow = (int32_t)P.long_order.size();
    P.long_lanes = opts ? opts->long_lanes : 0;
    size_t wide = 0;
    int64_t wide_nodes = 0;
    for (size_t b = 0; b < P.longs.size(); ++b)
      if (P.longs[b].maxw > kWarp) {
        P.long_order.push_back((int32_t)b);
        wide = std::max(wide, (size_t)(P.longs[b].nn + 2) * 8);
        wide_nodes += P.longs[b].nn;
      }
    // Team of a wide one: a block is faster on its own, warps fill the chip
    // better once there are many BDDs, the later the more nodes these have.
    // Path costs in shared memory while the blocks this leaves room for (at most
    // eight an SM, by their threads) are all of them.  us per iteration and per
    // iteration recorded and reversed, shared memory / scratch / warps:
    //   1,850 nodes a BDD: 608 BDDs 89, 372 / 97, 376 / 132, 492
    //                    1,520 BDDs 174, 811 / 184, 814 / 136, 678
    //   16,900 nodes:      152 BDDs 217, 1180 / 252, 1226 / 670, 3491
    //                      608 BDDs 1360, 3232 / 425, 1859 / 1236, 5092
    //                    3,648 BDDs - / 1469, 7278 / 1425, 6102
    //   71,000 nodes:    3,648 BDDs - / 4007, 21386 / 5965, 23425
    //                    4,864 BDDs - / 5303, 30087 / 6310, 25236
    const int64_t nwide = (int64_t)P.longs.size() - P.num_long_narrow;
    const int64_t fit = wide <= 200 * 1024 ? std::min<int64_t>(8, (int64_t)(227 * 1024 / (wide + 1024))) : 0;
    P.long_wide_smem = nwide <= kSms * fit ? (int32_t)wide : 0;
    P.long_wide_block = nwide <= kSms * std::min<int64_t>(24, 6 + (nwide ? wide_nodes / nwide : 0) / 1700);
  }
  const int64_t num_slots = slot_base;
  if (num_slots >= (int64_t)INT32_MAX || node_base >= (int64_t)INT32_MAX)
    return fail(DG_EINVAL, "dg_plan: arena exceeds 2^31 slots or nodes");

  // ---- 3. variable CSR (slots of each variable, rows ascending) -----------
  P.var_ptr.assign(n + 1, 0);
  for (int64_t s = 0; s < nnz; ++s) P.var_ptr[R->col[s] + 1]++;
  for (int32_t i = 0; i < n; ++i) P.var_ptr[i + 1] += P.var_ptr[i];
  P.var_slots.assign(nnz, 0);
  {
    std::vector<int32_t> cur(P.var_ptr.begin(), P.var_ptr.end() - 1);
    for (int64_t s = 0; s < nnz; ++s) P.var_slots[cur[R->col[s]]++] = (int32_t)slot_of_csr[s];
  }
  P.c.assign(R->c, R->c + n);
  P.var_ell.assign((size_t)kEll * n, -1);
  P.wide_vars.clear();
  for (int32_t i = 0; i < n; ++i) {
    const int d = P.var_ptr[i + 1] - P.var_ptr[i];
    for (int r = 0; r < std::min(d, kEll); ++r) P.var_ell[(size_t)r * n + i] = P.var_slots[P.var_ptr[i] + r];
    if (d > kEll) P.var_ell[(size_t)(kEll - 1) * n + i] = -2 - P.var_ell[(size_t)(kEll - 1) * n + i];
    if (d > kWide) P.wide_vars.push_back(i);
  }
  P.invdeg.assign(n, 0.0f);
  for (int32_t i = 0; i < n; ++i) {
    int d = P.var_ptr[i + 1] - P.var_ptr[i];
    P.invdeg[i] = d > 0 ? (float)(1.0 / d) : 0.0f;
  }
  // ---- 4. lower-bound chunks: per instance its rows, then its variables ----
  const int kChunk = 4096;
  P.inst_chunk_ptr.assign(ni + 1, 0);
  for (int k = 0; k < ni; ++k) {
    for (int kind = 0; kind < 2; ++kind) {
      int64_t b = kind == 0 ? P.inst_row_ptr[k] : P.inst_var_ptr[k];
      int64_t e = kind == 0 ? P.inst_row_ptr[k + 1] : P.inst_var_ptr[k + 1];
      for (int64_t x = b; x < e; x += kChunk) {
        P.lb_chunks.insert(P.lb_chunks.end(), {k, kind, (int32_t)x, (int32_t)std::min<int64_t>(e, x + kChunk)});
      }
    }
    P.inst_chunk_ptr[k + 1] = (int32_t)(P.lb_chunks.size() / 4);
  }
  // variables no row covers keep their cost: their term of the bound is the
  // constant min(0, c_i) (their S_i is an empty sum, 0, so the kernels may add
  // min(0, S_i) = 0 for them as for every other variable)
  P.inst_unc.assign(ni, 0.0);
  for (int k = 0; k < ni; ++k)
    for (int32_t i = P.inst_var_ptr[k]; i < P.inst_var_ptr[k + 1]; ++i)
      if (P.var_ptr[i + 1] == P.var_ptr[i]) P.inst_unc[k] += std::min(0.0, P.c[i]);
  const int num_chunks = (int)(P.lb_chunks.size() / 4);

  // ---- 5. arena offsets ----------------------------------------------------
  size_t o = 0;
  auto put = [&](size_t bytes) {
    size_t at = o;
    o = align_up(o + std::max<size_t>(bytes, 1), 256);
    return at;
  };
  P.off.tiles = put(P.tiles.size() * sizeof(Tile));
  P.off.unit_shapes = put(P.unit_shapes.size() * sizeof(UnitShape));
  P.off.unit_runs = put(P.unit_runs.size() * 2);
  P.off.desc = put(P.desc.size() * 2);
  P.off.lohi8 = put(P.lohi8.size() * 2);
  P.off.slot_var = put(num_slots * 4);
  P.off.slot_row = put(num_slots * 4);
  P.off.var_ptr = put((size_t)(n + 1) * 4);
  P.off.var_slots = put((size_t)nnz * 4);
  P.off.var_ell = put((size_t)kEll * n * 4);
  P.off.wide_vars = put(P.wide_vars.size() * 4);
  P.off.c = put((size_t)n * 8);
  P.off.invdeg = put((size_t)n * 4);
  P.off.inst_row_ptr = put((size_t)(ni + 1) * 8);
  P.off.inst_var_ptr = put((size_t)(ni + 1) * 4);
  P.off.lb_chunks = put((size_t)num_chunks * 16);
  P.off.inst_chunk_ptr = put((size_t)(ni + 1) * 4);
  P.off.inst_unc = put((size_t)ni * 8);
  P.off.longs = put(P.longs.size() * sizeof(LongBdd));
  P.off.long_code = put(P.long_code.size() * sizeof(int2));
  P.off.long_lvl = put(P.long_lvl.size() * 4);
  P.off.long_in_ptr = put(P.long_in_ptr.size() * 4);
  P.off.long_in = put(P.long_in.size() * 4);
  P.off.long_order = put(P.long_order.size() * 4);
  P.off.long_items = put(P.long_items.size() * sizeof(LongItem));
  P.off.S = put((size_t)n * 4);
  P.off.var_avg = put((size_t)n * 4);
  P.off.slot_avg = put((size_t)num_slots * 4);
  P.off.E = put((size_t)m * 4);
  P.off.lb_part = put((size_t)num_chunks * 8);
  P.off.long_d = put((size_t)P.long_cost_size * 4);
  P.off.long_t = put((size_t)P.long_cost_size * 4);
  P.off.nodecost = put(P.lohi8.size() * 4);
  P.off.slot_invdeg = put((size_t)num_slots * 4);
  P.off.total = o;
  P.smem_sweep = align_up(smem_max, 16);
  P.smem_adjoint = align_up(smem_adj_max, 16);

  dg_sizes& z = P.sizes;
  z.arena_bytes = P.off.total;
  z.num_slots = num_slots;
  z.num_lambda = nnz;
  z.num_nodes = num_nodes;
  z.num_nodes_padded = node_base;
  z.n = n;
  z.m = m;
  z.num_inst = ni;
  z.num_tiles = T;
  z.max_hops = max_hops;
  z.max_width = max_width;
  z.smem_bytes = P.smem_sweep;
  z.num_launch_groups = (int32_t)P.groups.size();
  z.num_long_bdds = (int64_t)P.longs.size();
  z.num_long_nodes = num_long_nodes;
  return DG_OK;
}

// Structural invariants of the arena image, checked on the host (the kernels
// index shared and global memory with these numbers without bounds checks).
dg_status validate_plan(const Plan& P) {
  auto bad = [](const std::string& m) { return fail(DG_EINVAL, "dg_plan_validate: " + m); };
  const int32_t n = P.sizes.n;
  const int64_t m = P.sizes.m, NS = P.sizes.num_slots, NL = P.sizes.num_lambda;
  const int64_t T = (int64_t)P.tiles.size();
  if ((int64_t)P.desc.size() != NS || (int64_t)P.slot_var.size() != NS || (int64_t)P.slot_row.size() != NS ||
      (int64_t)P.slot_to_csr.size() != NS || (int64_t)P.lohi8.size() != P.sizes.num_nodes_padded)
    return bad("array sizes disagree with the plan sizes");
  // unit shapes: window, states and runs in range
  for (const UnitShape& s : P.unit_shapes) {
    if (s.W < 2 || s.W > kUnitMaxW || s.W % 2 != 0 || s.k < 1 || s.start < 0 || s.start >= s.W || s.accept <= 0 ||
        s.accept >= (1 << s.W) || s.nruns < 1 || s.run_base < 0 ||
        (size_t)s.run_base + (size_t)s.nruns > P.unit_runs.size())
      return bad("unit shape out of range");
    int prev = 0, rows = -1;
    for (int r = 0; r < s.nruns; ++r) {
      const int e = P.unit_runs[s.run_base + r] >> 2;
      if (e <= prev || e > s.k) return bad("unit shape runs not ascending");
      rows += (e - prev + 1) / 2;
      prev = e;
    }
    int types = 0;
    for (int h = 0, r = 0; unit_short(s) && h < s.k; ++h) {
      if (h >= (P.unit_runs[s.run_base + r] >> 2)) ++r;
      types |= (P.unit_runs[s.run_base + r] & 3) << (2 * h);
    }
    if (prev != s.k || rows != s.rows || types != s.types) return bad("unit shape runs do not cover its levels");
  }
  // tiles: contiguous bases, sane shapes, every lane's BDD well formed
  int64_t node_base = 0, slot_base = 0, real_nodes = 0, real_slots = 0;
  std::vector<int64_t> csr_seen(NL, 0);
  for (int64_t t = 0; t < T; ++t) {
    const Tile& tl = P.tiles[t];
    const std::string at = "tile " + std::to_string(t) + ": ";
    if (tl.node_base != node_base || tl.slot_base != slot_base) return bad(at + "bases not contiguous");
    if (tl.nbdd < 1 || tl.nbdd > kWarp || tl.nhops < 1 || tl.nmax < 3 || tl.nmax > kMaxNodesPerBdd + 2 ||
        tl.maxw < 1 || tl.maxw > kMaxWidth || tl.ring != ring_size(tl.maxw))
      return bad(at + "shape out of range");
    if (tl.unit < 0 || tl.unit > (int32_t)P.unit_shapes.size() ||
        (tl.unit && (P.unit_shapes[tl.unit - 1].k != tl.nhops || slot_base >= P.unit_slots)) ||
        (!tl.unit && slot_base < P.unit_slots))
      return bad(at + "unit shape does not fit the tile");
    for (int b = 0; b < kWarp; ++b) {
      int first = 2, level_w = 0, last_h = -1, row = -1;
      for (int h = 0; h < tl.nhops; ++h) {
        const int64_t q = slot_base + (int64_t)h * kWarp + b;
        const int f = P.desc[q] & 0xFF, w = P.desc[q] >> 8;
        if (b >= tl.nbdd || last_h >= 0) {
          if (P.desc[q] != 0 || P.slot_var[q] != -1 || P.slot_to_csr[q] != -1)
            return bad(at + "padding slot in use");
          continue;
        }
        if (w == 0) {
          if (h == 0) return bad(at + "lane without a BDD");
          last_h = h - 1;
          if (P.slot_var[q] != -1 || P.slot_to_csr[q] != -1) return bad(at + "padding slot in use");
          continue;
        }
        if (f != first || (h == 0 && w != 1) || w > tl.maxw || f + w > tl.nmax)
          return bad(at + "level descriptor inconsistent");
        if (P.slot_var[q] < 0 || P.slot_var[q] >= n) return bad(at + "variable id out of range");
        if (row < 0) row = P.slot_row[q];
        if (P.slot_row[q] != row || row < 0 || row >= m) return bad(at + "slot rows of a lane differ");
        const int64_t c = P.slot_to_csr[q];
        if (c < 0 || c >= NL || csr_seen[c]++) return bad(at + "slot map not a bijection");
        first = f + w;
        level_w = w;
        real_slots++;
        real_nodes += w;
      }
      if (b >= tl.nbdd) continue;
      if (last_h < 0) last_h = tl.nhops - 1;
      if (tl.unit && last_h != tl.nhops - 1) return bad(at + "unit tile lane with fewer levels");
      // a unit tile's lanes are sweeped by its shape alone: nodes as states
      std::vector<int> state(1, tl.unit ? P.unit_shapes[tl.unit - 1].start : 0), next;
      const uint16_t* run = tl.unit ? &P.unit_runs[P.unit_shapes[tl.unit - 1].run_base] : nullptr;
      // children: next level's nodes (no level skipped) or the bottom; the
      // last level only the terminals; at least one child not the bottom
      int f = 2;
      for (int h = 0; h <= last_h; ++h) {
        const int64_t q = slot_base + (int64_t)h * kWarp + b;
        const int w = P.desc[q] >> 8;
        const int fn = f + w;
        const int wn = h < last_h ? (P.desc[q + kWarp] >> 8) : 0;
        for (int r = 0; r < w; ++r) {
          const uint32_t code = P.lohi8[node_base + (int64_t)(f + r - 2) * kWarp + b];
          const uint32_t ch[2] = {code & 0xFFu, code >> 8};
          if (ch[0] == (uint32_t)kBotCode && ch[1] == (uint32_t)kBotCode) return bad(at + "node with no path to top");
          for (uint32_t c : ch) {
            const bool term = c == (uint32_t)kTopCode || c == (uint32_t)kBotCode;
            if (h == last_h ? !term : (c == (uint32_t)kTopCode || (!term && (c < (uint32_t)fn || c >= (uint32_t)(fn + wn)))))
              return bad(at + "child code outside the next level");
          }
        }
        if (tl.unit) {
          const UnitShape& s = P.unit_shapes[tl.unit - 1];
          if (h >= (*run >> 2)) ++run;
          next.assign(wn, -1);
          for (int r = 0; r < w; ++r) {
            const uint32_t code = P.lohi8[node_base + (int64_t)(f + r - 2) * kWarp + b];
            const int u = state[r];
            if (u < 0 || (r > 0 && u >= state[r - 1])) return bad(at + "unit states not descending");
            for (int beta = 0; beta < 2; ++beta) {
              const uint32_t c = beta ? code >> 8 : code & 0xFFu;
              if (c == (uint32_t)kBotCode) continue;
              const int to = beta ? unit_o(*run & 3, u) : unit_z(*run & 3, u);
              if (to < 0 || to >= s.W) return bad(at + "unit state outside the window");
              if (c == (uint32_t)kTopCode) {
                if (!((s.accept >> to) & 1)) return bad(at + "unit state not accepted");
              } else if (next[c - fn] >= 0 && next[c - fn] != to) {
                return bad(at + "unit states of a node differ");
              } else {
                next[c - fn] = to;
              }
            }
          }
          state.swap(next);
        }
        f = fn;
      }
      (void)level_w;
    }
    node_base += (int64_t)(tl.nmax - 2) * kWarp;
    slot_base += (int64_t)tl.nhops * kWarp;
  }
  if (node_base != P.sizes.num_nodes_padded || slot_base != P.long_slot_base) return bad("tiles do not cover the arrays");
  // long BDDs: consecutive slot ranges after the tiles, levels and children
  // consistent, in-arc lists exactly the arcs into each node in (parent,
  // beta) order
  {
    int64_t lslot = P.long_slot_base, code_base = 0, lvl_base = 0, cost_base = 0;
    for (size_t b = 0; b < P.longs.size(); ++b) {
      const LongBdd& L = P.longs[b];
      const std::string at = "long BDD " + std::to_string(b) + ": ";
      if (L.slot_base != lslot || L.code_base != code_base || L.lvl_base != lvl_base || L.cost_base != cost_base ||
          L.k < 1 || L.nn < 1 || L.row < 0 || L.row >= m || P.long_of_row[L.row] != (int32_t)b)
        return bad(at + "bases or shape inconsistent");
      const int32_t* lvl = P.long_lvl.data() + L.lvl_base;
      if ((size_t)(L.lvl_base + L.k + 1) > P.long_lvl.size() || lvl[0] != 2 || lvl[1] != 3 || lvl[L.k] != L.nn + 2)
        return bad(at + "level table inconsistent");
      const int64_t tslots = ((int64_t)L.k + kWarp - 1) / kWarp * kWarp;
      int row = -1;
      for (int64_t q = lslot; q < lslot + tslots; ++q) {
        const int h = (int)(q - lslot);
        if (h >= L.k) {
          if (P.slot_var[q] != -1 || P.slot_to_csr[q] != -1) return bad(at + "padding slot in use");
          continue;
        }
        if (lvl[h + 1] <= lvl[h]) return bad(at + "empty level");
        if (P.slot_var[q] < 0 || P.slot_var[q] >= n) return bad(at + "variable id out of range");
        if (row < 0) row = P.slot_row[q];
        if (P.slot_row[q] != row || row != L.row) return bad(at + "slot rows differ");
        const int64_t c = P.slot_to_csr[q];
        if (c < 0 || c >= NL || csr_seen[c]++) return bad(at + "slot map not a bijection");
        real_slots++;
      }
      real_nodes += L.nn;
      std::vector<int32_t> indeg(L.nn + 2, 0);
      for (int h = 0; h < L.k; ++h)
        for (int v = lvl[h]; v < lvl[h + 1]; ++v) {
          const int2 c = P.long_code[L.code_base + v - 2];
          if (c.x == (int)kBotCode && c.y == (int)kBotCode) return bad(at + "node with no path to top");
          for (int ch : {c.x, c.y}) {
            const bool term = ch == (int)kTopCode || ch == (int)kBotCode;
            const bool in_next = h + 1 < L.k && ch >= lvl[h + 1] && ch < lvl[h + 2];
            if (h + 1 == L.k ? !term : !(ch == (int)kBotCode || in_next)) return bad(at + "child outside the next level");
            if (ch >= 2) indeg[ch]++;
          }
        }
      for (int v = 2; v < L.nn + 2; ++v) {
        const int32_t b0 = P.long_in_ptr[L.code_base + v - 2], b1 = P.long_in_ptr[L.code_base + v - 1];
        if (b1 - b0 != indeg[v] || (v > 2 && indeg[v] == 0)) return bad(at + "in-arc list size wrong");
        int32_t prev = -1;
        for (int32_t i = b0; i < b1; ++i) {
          const int32_t e = P.long_in[i], par = e >> 1;
          if (e <= prev || par < 2 || par >= v) return bad(at + "in-arc list not ascending");
          const int2 c = P.long_code[L.code_base + par - 2];
          if ((e & 1 ? c.y : c.x) != v) return bad(at + "in-arc is not an arc");
          prev = e;
        }
      }
      lslot += tslots;
      code_base += L.nn;
      lvl_base += L.k + 1;
      cost_base += L.nn + 2;
    }
    if (lslot != NS || cost_base != P.long_cost_size || code_base != P.sizes.num_long_nodes)
      return bad("long BDDs do not cover the arrays");
    // the order list: a permutation, the narrow BDDs (levels within a warp) first
    if (P.long_order.size() != P.longs.size() || P.num_long_narrow < 0 ||
        P.num_long_narrow > (int32_t)P.longs.size())
      return bad("long BDD order malformed");
    if (P.long_lanes < 0 || P.long_lanes > kWarp || (P.long_lanes & (P.long_lanes - 1)) != 0)
      return bad("lanes per narrow long BDD not a power of two up to 32");
    std::vector<char> listed(P.longs.size(), 0);
    for (size_t i = 0; i < P.long_order.size(); ++i) {
      const int32_t b = P.long_order[i];
      if (b < 0 || b >= (int32_t)P.longs.size() || listed[b]++) return bad("long BDD order not a permutation");
      if ((P.longs[b].maxw <= kWarp) != ((int32_t)i < P.num_long_narrow))
        return bad("long BDD order: narrow and wide BDDs mixed");
    }
    // the unit ones: every item's BDDs have its shape, state for node
    if (P.num_long_unit < 0 || P.num_long_unit > P.num_long_narrow) return bad("long unit BDDs not narrow");
    std::vector<char> in_item(P.num_long_unit, 0);
    for (const LongItem& it : P.long_items) {
      if (it.G < 2 || it.G > kLongUnitMaxW || (it.G & (it.G - 1)) != 0 || it.nseg < 1 ||
          it.nseg > (it.G <= kUnitMaxW ? kWarp : kWarp / it.G) ||
          it.first < 0 || it.first + it.nseg > P.num_long_unit || it.start < 0 || it.start >= it.G || it.nruns < 1 ||
          it.run_base < 0 || (size_t)it.run_base + (size_t)it.nruns > P.unit_runs.size() ||
          long_unit_bytes(it.nseg, it.G, it.kmax, 0) > (size_t)P.long_unit_smem[0] ||
          long_unit_bytes(it.nseg, it.G, it.kmax, 1) > (size_t)P.long_unit_smem[1] ||
          long_unit_adjoint_bytes(it.nseg, it.kmax) > (size_t)P.long_unit_adj_smem)
        return bad("long unit item out of range");
      for (int x = it.first; x < it.first + it.nseg; ++x) {
        const LongBdd& L = P.longs[P.long_order[x]];
        if (in_item[x]++ || L.k > it.kmax) return bad("long unit item lists a BDD twice or too long a one");
        const int32_t* lvl = P.long_lvl.data() + L.lvl_base;
        std::vector<int> state(1, it.start), next;
        const uint16_t* run = &P.unit_runs[it.run_base];
        int left = it.nruns;
        for (int h = 0; h < L.k; ++h) {
          if (left > 1 && h >= (*run >> 2)) {
            ++run;
            --left;
          }
          next.assign(h + 1 < L.k ? lvl[h + 2] - lvl[h + 1] : 0, -1);
          for (int v = lvl[h]; v < lvl[h + 1]; ++v) {
            const int u = state[v - lvl[h]];
            if (u < 0 || (v > lvl[h] && u >= state[v - lvl[h] - 1])) return bad("long unit states not descending");
            const int2 cc = P.long_code[L.code_base + v - 2];
            for (int beta = 0; beta < 2; ++beta) {
              const int c = beta ? cc.y : cc.x;
              if (c == (int)kBotCode) continue;
              const int to = beta ? unit_o(*run & 3, u) : unit_z(*run & 3, u);
              if (to < 0 || to >= it.G) return bad("long unit state outside the window");
              if (c == (int)kTopCode) {
                if (!((it.accept >> to) & 1)) return bad("long unit state not accepted");
              } else if (next[c - lvl[h + 1]] >= 0 && next[c - lvl[h + 1]] != to) {
                return bad("long unit states of a node differ");
              } else {
                next[c - lvl[h + 1]] = to;
              }
            }
          }
          state.swap(next);
        }
        if (left > 1) return bad("long unit item's BDD shorter than its runs");
      }
    }
    for (char c : in_item)
      if (!c) return bad("long unit BDD in no item");
    if (P.long_plain != 0 && P.long_plain != P.num_long_unit) return bad("long BDDs of the plain sweeps malformed");
  }
  if (real_slots != NL || real_nodes != P.sizes.num_nodes) return bad("slot or node count mismatch");
  // variables: CSR and ELL columns point back at their own slots, rows ascending
  if ((int64_t)P.var_ptr.size() != (int64_t)n + 1 || P.var_ptr[0] != 0 || P.var_ptr[n] != NL)
    return bad("variable pointers malformed");
  size_t next_wide = 0;
  for (int32_t i = 0; i < n; ++i) {
    if (P.var_ptr[i + 1] < P.var_ptr[i]) return bad("variable pointers not monotone");
    int prev_row = -1;
    for (int32_t k = P.var_ptr[i]; k < P.var_ptr[i + 1]; ++k) {
      const int32_t q = P.var_slots[k];
      if (q < 0 || q >= NS || P.slot_var[q] != i) return bad("variable " + std::to_string(i) + ": slot list wrong");
      if (P.slot_row[q] <= prev_row) return bad("variable " + std::to_string(i) + ": rows not ascending");
      prev_row = P.slot_row[q];
    }
    const int d = P.var_ptr[i + 1] - P.var_ptr[i];
    for (int r = 0; r < kEll; ++r) {
      int32_t e = P.var_ell[(size_t)r * n + i];
      if (d > kEll && r == kEll - 1) {
        if (e > -2) return bad("variable " + std::to_string(i) + ": ELL overflow mark missing");
        e = -2 - e;
      }
      const int32_t want = r < d ? P.var_slots[P.var_ptr[i] + r] : -1;
      if (e != want) return bad("variable " + std::to_string(i) + ": ELL column disagrees with the slot list");
    }
    if (d > kWide) {
      if (next_wide >= P.wide_vars.size() || P.wide_vars[next_wide] != i)
        return bad("variable " + std::to_string(i) + ": missing from the wide-variable list");
      ++next_wide;
    }
  }
  if (next_wide != P.wide_vars.size()) return bad("wide-variable list lists a narrow variable");
  // launch groups cover the tiles in order
  int32_t t0 = 0;
  for (const LaunchGroup& g : P.groups) {
    if (g.tile0 != t0 || g.tile1 <= g.tile0 || g.stream < 0 || g.stream >= kStreams) return bad("launch groups malformed");
    for (int32_t t = g.tile0; t < g.tile1; ++t) {
      const Tile& tl = P.tiles[t];
      if (tl.unit ? g.unit_w < P.unit_shapes[tl.unit - 1].W ||
                        (g.unit_short && !unit_short(P.unit_shapes[tl.unit - 1])) ||
                        (size_t)g.unit_bytes1 < unit_smem_bytes(P.unit_shapes[tl.unit - 1], 1) ||
                        (size_t)g.unit_bytes0 < unit_smem_bytes(P.unit_shapes[tl.unit - 1], 0)
                  : g.unit_w != 0)
        return bad("launch group " + std::to_string(t0) + ": does not fit its unit tiles");
      if ((size_t)g.region_bytes < sweep_smem_bytes(tl.nmax, tl.nhops, 1, tl.ring) ||
          (size_t)g.region_bwd1 < sweep_smem_bytes_bwd(tl.nmax, tl.nhops, 1) ||
          g.meta_bytes < (tl.nmax - 2) * kWarp * 2)
        return bad("launch group " + std::to_string(t0) + ": shared memory smaller than a tile needs");
    }
    t0 = g.tile1;
  }
  if (t0 != T) return bad("launch groups do not cover the tiles");
  // a chain launches the kernels of the unit rows alone
  if (P.chained) {
    if (P.long_plain != (int32_t)P.longs.size()) return bad("chained launches with other long BDDs");
    for (const LaunchGroup& g : P.groups)
      if (g.unit_w == 0) return bad("chained launches with mixed tiles");
  }
  // bound chunks: per instance its rows, then its variables, in order
  const int ni = P.sizes.num_inst;
  for (int k = 0; k < ni; ++k) {
    int64_t rows_at = P.inst_row_ptr[k], vars_at = P.inst_var_ptr[k];
    for (int32_t c = P.inst_chunk_ptr[k]; c < P.inst_chunk_ptr[k + 1]; ++c) {
      const int32_t* ch = &P.lb_chunks[(size_t)c * 4];
      if (ch[0] != k || ch[3] <= ch[2]) return bad("bound chunk malformed");
      int64_t& at = ch[1] == 0 ? rows_at : vars_at;
      if (ch[2] != at) return bad("bound chunks leave a gap");
      at = ch[3];
    }
    if (rows_at != P.inst_row_ptr[k + 1] || vars_at != P.inst_var_ptr[k + 1]) return bad("bound chunks do not cover an instance");
  }
  return DG_OK;
}

}  // namespace dg
