// Host-only check of the sweep kernel's work lists (sweep_plan, sweep_plan_batch
// over the subsets of a batch, sweep_plan_cross over the rows and the panel columns
// of a serving step), built by tests/test_sweep_plan.py with nvcc and run on the
// CPU: no device call.  For every list it checks that
//   - every block of each triangle (rows in pairs, from the diagonal to the right
//     edge), or of each row pair and panel block, is covered once over the stages
//     of all four sweeps;
//   - a tile covered by several items is in the list of split tiles with one
//     part slot per item and product it touches, all slots used exactly once, and
//     no more slots than the serving engine has room for;
//   - items stay inside the triangle or the ranges, and the waves of whole tiles
//     have one tile per cluster.
// Prints one line per failure and "checked N lists, F failures".
#include "../paper_1410_4803_gb300/csrc/ibs_sweep.cu"

#include <cmath>
#include <map>
#include <random>
#include <set>
#include <tuple>
#include <utility>

namespace {

int failures = 0;
void fail(const char* what, int64_t n, int64_t m, int c) {
  ++failures;
  printf("FAIL %s: n=%lld m=%lld clusters=%d\n", what, (long long)n, (long long)m, c);
}

using Tile = std::tuple<int, int, int>;  // subset, I, J

// What a list has to cover of a subset: its blocks (row pair, column), over 4 * stages stages.
struct Want {
  int stages;
  std::set<std::pair<int, int>> blocks;
};

Want triangle(int64_t n, int64_t m) {
  Want w{ibs::sweep_stages(m), {}};
  const int T = (int)((n + 127) / 128);
  for (int I = 0; I < T; I += 2)
    for (int J = I; J < T; ++J) w.blocks.insert({I, J});
  return w;
}

// (n, m: for the messages)
void check(const ibs::SweepPlan& p, const std::vector<Want>& want, int64_t n, int64_t m, int C, bool one) {
  using namespace ibs;
  std::map<Tile, std::vector<std::pair<int, int>>> cover;
  std::map<Tile, SweepGroup> groups;
  std::vector<int> used((size_t)p.slots, 0), wave((size_t)p.waves, 0);
  for (const SweepGroup& g : p.groups) groups[{g.subset, g.I, g.J}] = g;
  if (p.clusters < 1 || p.clusters > C || p.first.size() != (size_t)C + 1) fail("cluster count", n, m, C);
  if (one && p.slots > sweep_max_slots(C)) fail("slots", n, m, C);
  for (const SweepItem& it : p.items) {
    if (it.subset < 0 || it.subset >= (int)want.size()) {
      fail("subset", n, m, C);
      continue;
    }
    const Want& w = want[(size_t)it.subset];
    const int S = w.stages;
    if (it.w < 1 || it.w > 3 || it.q0 < 0 || it.q1 <= it.q0 || it.q1 > 4 * S) fail("item", n, m, C);
    for (int b = 0; b < it.w; ++b) {
      if (w.blocks.count({it.I, it.J + b}) == 0) fail("item outside", n, m, C);
      cover[{it.subset, it.I, it.J + b}].push_back({it.q0, it.q1});
    }
    if (it.wave >= 0) {
      if (it.wave >= p.waves || it.slot >= 0) fail("wave", n, m, C);
      else ++wave[(size_t)it.wave];
    }
    if (it.slot < 0) {
      if (it.q0 != 0 || it.q1 != 4 * S || !p.scratch) fail("whole tile", n, m, C);
      continue;
    }
    const auto g = groups.find({it.subset, it.I, it.J});
    if (g == groups.end()) {
      fail("split tile without a group", n, m, C);
      continue;
    }
    int slot = it.slot, base = g->second.slot;
    for (int pr = 0; pr < 3; ++pr) {
      const int a = pr * S, b = pr == 2 ? 4 * S : a + S;
      if (it.q0 < b && it.q1 > a) {
        if (slot < base || slot >= base + g->second.pieces[pr] || used[(size_t)slot]++) fail("part slot", n, m, C);
        ++slot;
      }
      base += g->second.pieces[pr];
    }
  }
  // one matrix or step: whole tiles in waves only, where the others have slots; and
  // no cluster with twice its share of the work
  if (one) {
    std::set<std::pair<int, int>> rest;
    bool whole = false;
    double most = 0, total = 0;
    for (int c = 0; c < p.clusters; ++c) {
      double load = 0;
      for (int i = p.first[(size_t)c]; i < p.first[(size_t)c + 1]; ++i) {
        const SweepItem& it = p.items[(size_t)i];
        load += stage_cost(it.w) * (it.q1 - it.q0);
        if (it.wave < 0) {
          rest.insert({it.I, it.J});
          whole |= it.slot < 0;
        }
      }
      most = std::max(most, load);
      total += load;
    }
    if (whole && 3 * (int)rest.size() + C <= sweep_max_slots(C)) fail("whole tile outside the waves", n, m, C);
    if (most > 2 * total / p.clusters + 8 * 620) fail("balance", n, m, C);
  }
  for (int u : used)
    if (u != 1) fail("unused slot", n, m, C);
  for (int u : wave)
    if (u != C) fail("wave size", n, m, C);
  for (size_t k = 0; k < want.size(); ++k)
    for (const auto& b : want[k].blocks) {
      auto v = cover[{(int)k, b.first, b.second}];
      std::sort(v.begin(), v.end());
      int e = 0;
      for (const auto& r : v) {
        if (r.first != e) fail("stages not contiguous", n, m, C);
        e = r.second;
      }
      if (e != 4 * want[k].stages) fail("stages not covered", n, m, C);
    }
}

// Rows of `rows` blocks against panel blocks [at, at + len), wrapping around at `panel`.
void check_cross(int64_t panel, int64_t rows, int64_t at, int64_t len, int64_t m, int C) {
  const int64_t end = at + len;
  const int64_t cols[2][2] = {{at, std::min(end, panel)}, {0, std::max<int64_t>(0, end - panel)}};
  Want w{ibs::sweep_stages(m), {}};
  for (const auto& r : cols)
    for (int64_t J = r[0]; J < r[1]; ++J)
      for (int64_t I = 0; I < rows; I += 2) w.blocks.insert({(int)I, (int)J});
  check(ibs::sweep_plan_cross(rows, cols, m, C), {w}, panel, m, C, true);
}

// Steps of serving: whole tiles up to the last, no block more than is needed,
// one step for a lone request of one or two blocks over up to 155,000 samples
// (76 clusters), no more steps over a panel than the shortest allowed length gives.
void check_steps(int64_t panel, int64_t rows, int c) {
  using namespace ibs;
  const int64_t pairs = (rows + 1) / 2;
  int64_t steps = 0, left = panel;
  for (; left > 0; ++steps) {
    const int64_t len = sweep_step_blocks(panel, rows, left, c);
    if (len < 1 || len > left || (len < left && len % 3 != 0)) return fail("step length", panel, rows, c);
    left -= len;
  }
  if (pairs == 1 && panel <= 16 * c && steps != 1) fail("steps of a lone request", panel, rows, c);
  if (steps > std::max<int64_t>(33, panel * pairs / (8 * c) + 2)) fail("steps over the panel", panel, rows, c);
}

}  // namespace

int main() {
  int lists = 0;
  for (int64_t n : {1, 63, 64, 128, 129, 256, 257, 384, 385, 700, 1501, 3000, 4096, 5000, 9999, 20000})
    for (int64_t m : {1, 288, 289, 577, 1000, 1500, 30011, 100000, 500000, 2097151})
      for (int c : {1, 5, 74, 76}) {
        check(ibs::sweep_plan(n, m, c), {triangle(n, m)}, n, m, c, true);
        ++lists;
      }
  std::mt19937 g(1);
  for (int rep = 0; rep < 60; ++rep) {
    std::vector<std::pair<int64_t, int64_t>> shapes(1 + g() % 40);
    for (auto& s : shapes) s = {1 + g() % (rep % 3 ? 3000 : 300), 1 + g() % (rep % 5 ? 80000 : 2000)};
    std::vector<Want> want;
    for (const auto& s : shapes) want.push_back(triangle(s.first, s.second));
    for (int c : {5, 76}) {
      check(ibs::sweep_plan_batch(shapes, c), want, shapes[0].first, shapes[0].second, c, false);
      ++lists;
    }
  }
  for (int rep = 0; rep < 400; ++rep) {
    // up to the 32 blocks of 4,096 rows; panels of up to 100,000 samples
    const int64_t panel = 1 + (int64_t)std::exp((double)(g() % 1000) / 1000 * std::log(782.0)), rows = 1 + g() % 32;
    const int64_t m = 1 + (int64_t)std::exp((double)(g() % 1000) / 1000 * std::log(rep % 10 ? 60000.0 : 2000000.0));
    const int c = rep % 8 == 0 ? 1 + (int)(g() % 80) : 76;
    const int64_t at = g() % panel, left = rep % 3 ? panel : 1 + g() % panel;
    check_cross(panel, rows, at, ibs::sweep_step_blocks(panel, rows, left, c), m, c);
    check_cross(panel, rows, 0, panel, m, c);  // the unbatched path: the whole panel
    lists += 2;
  }
  for (int64_t rows = 0; rows <= 18; ++rows)  // serving steps on the panel's code bits
    for (int64_t n : {int64_t{300}, int64_t{20000}, int64_t{20001}, int64_t{2147483647}}) {
      const bool small = n <= 20000;  // panels of 20,000 markers
      if (ibs::few_rows_pay(rows, n, 20000) != (rows >= 1 && (rows <= 8 || (small && rows <= 16))))
        fail("few rows", n, rows, 0);
    }
  for (int64_t panel : {1, 2, 3, 4, 40, 156, 157, 607, 608, 609, 782, 1215, 1216, 1217, 1563, 16384})
    for (int64_t rows = 1; rows <= 32; ++rows)
      for (int c : {1, 5, 76}) check_steps(panel, rows, c);
  printf("checked %d lists, %d failures\n", lists, failures);
  return failures == 0 ? 0 : 1;
}
