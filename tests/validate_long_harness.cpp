// Host-only harness for the plan validator on long rows: builds the plan of a
// few rows of +1s and of a general one next to a short row, then corrupts one
// invariant at a time and prints, per case, the status and message of
// validate_plan.  Compiled and run by tests/test_lib_cpu.py together with
// builder.cpp; it supplies the error-reporting functions that api.cu defines in
// the library.
#include <cstdio>
#include <functional>
#include <string>
#include <vector>

#include "dg_internal.h"

namespace dg {
static std::string g_msg;
dg_status fail(dg_status st, const std::string& msg) {
  g_msg = msg;
  return st;
}
void clear_error() { g_msg.clear(); }
}  // namespace dg

int main() {
  using namespace dg;
  // sum of k <= 1 for k = 300, 280 (long, two states), the same with coefficient
  // 2, sum of 60 = 12 (long, 13 states), and one short row
  const int n = 300;
  const int len[] = {300, 280, 300, 60, 3}, coefs[] = {1, 1, 2, 1, 1}, rhs_of[] = {1, 1, 2, 12, 1};
  const int8_t sense[] = {0, 0, 0, 2, 0};
  std::vector<int64_t> row_ptr = {0};
  std::vector<int32_t> col, coef, rhs;
  for (int j = 0; j < 5; ++j) {
    for (int i = 0; i < len[j]; ++i) {
      col.push_back(i);
      coef.push_back(coefs[j]);
    }
    row_ptr.push_back((int64_t)col.size());
    rhs.push_back(rhs_of[j]);
  }
  std::vector<double> c(n, 1.0);
  dg_rows R{};
  R.num_inst = 1;
  R.n = n;
  R.m = 5;
  R.row_ptr = row_ptr.data();
  R.col = col.data();
  R.coef = coef.data();
  R.sense = sense;
  R.rhs = rhs.data();
  R.c = c.data();
  dg_options o{};
  o.long_lanes = 1;  // the two rows of two states to one warp
  Plan P;
  if (build_plan(&R, &o, P) != DG_OK) {
    std::printf("build failed: %s\n", g_msg.c_str());
    return 1;
  }
  auto run = [&](const char* name, const std::function<void(Plan&)>& corrupt) {
    Plan Q = P;
    corrupt(Q);
    g_msg.clear();
    const dg_status st = validate_plan(Q);
    std::printf("%s|%d|%s\n", name, (int)st, g_msg.c_str());
  };
  run("intact", [](Plan&) {});
  run("order_out_of_range", [](Plan& Q) { Q.long_order[0] = 1 << 28; });
  run("order_negative", [](Plan& Q) { Q.long_order[0] = -(1 << 28); });
  run("order_duplicate", [](Plan& Q) { Q.long_order[0] = Q.long_order[1]; });
  run("item_first", [](Plan& Q) { Q.long_items[0].first += 1; });
  run("item_levels", [](Plan& Q) { Q.long_items[0].kmax -= 1; });
  run("item_count", [](Plan& Q) { Q.long_items[0].nseg = 1; });
  run("item_start", [](Plan& Q) { Q.long_items[0].start = Q.long_items[0].G; });
  run("item_runs", [](Plan& Q) { Q.long_items[0].run_base = (int32_t)Q.unit_runs.size(); });
  run("item_memory", [](Plan& Q) { Q.long_unit_smem[1] = 0; });
  run("plain_from", [](Plan& Q) { Q.long_plain = 1; });
  run("chained", [](Plan& Q) { Q.chained = true; });
  return 0;
}
