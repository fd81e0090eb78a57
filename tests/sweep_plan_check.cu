// Host-only check of the sweep kernel's work lists (sweep_plan, and sweep_plan_batch over the subsets of a
// batch), built by
// tests/test_sweep_plan.py with nvcc and run on the CPU: no device call.  For
// every list it checks that
//   - every block of each triangle (rows in pairs, from the diagonal to the right
//     edge) is covered once over the stages of all four sweeps;
//   - a tile covered by several items is in the list of split tiles with one
//     part slot per item and product it touches, all slots used exactly once;
//   - items stay inside the triangle, and the waves of whole tiles have one tile
//     per cluster.
// Prints one line per failure and "checked N lists, F failures".
#include "../paper_1410_4803_gb300/csrc/ibs_sweep.cu"

#include <map>
#include <random>
#include <tuple>
#include <utility>

namespace {

int failures = 0;
void fail(const char* what, int64_t n, int64_t m, int c) {
  ++failures;
  printf("FAIL %s: n=%lld m=%lld clusters=%d\n", what, (long long)n, (long long)m, c);
}

using Tile = std::tuple<int, int, int>;  // subset, I, J

void check(const ibs::SweepPlan& p, const std::vector<std::pair<int64_t, int64_t>>& shapes, int C) {
  using namespace ibs;
  const int64_t n = shapes[0].first, m = shapes[0].second;  // (for the messages)
  std::map<Tile, std::vector<std::pair<int, int>>> cover;
  std::map<Tile, SweepGroup> groups;
  std::vector<int> used((size_t)p.slots, 0), wave((size_t)p.waves, 0);
  for (const SweepGroup& g : p.groups) groups[{g.subset, g.I, g.J}] = g;
  if (p.clusters < 1 || p.clusters > C || p.first.size() != (size_t)C + 1) fail("cluster count", n, m, C);
  for (const SweepItem& it : p.items) {
    if (it.subset < 0 || it.subset >= (int)shapes.size()) {
      fail("subset", n, m, C);
      continue;
    }
    const int T = (int)((shapes[(size_t)it.subset].first + 127) / 128), S = sweep_stages(shapes[(size_t)it.subset].second);
    if (it.w < 1 || it.w > 3 || it.I % 2 || it.I < 0 || it.J < it.I || it.J + it.w > T || it.q0 < 0 || it.q1 <= it.q0 ||
        it.q1 > 4 * S)
      fail("item", n, m, C);
    for (int b = 0; b < it.w; ++b) cover[{it.subset, it.I, it.J + b}].push_back({it.q0, it.q1});
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
  for (int u : used)
    if (u != 1) fail("unused slot", n, m, C);
  for (int u : wave)
    if (u != C) fail("wave size", n, m, C);
  size_t blocks = 0;
  for (size_t k = 0; k < shapes.size(); ++k) {
    const int T = (int)((shapes[k].first + 127) / 128), S = sweep_stages(shapes[k].second);
    for (int I = 0; I < T; I += 2)
      for (int J = I; J < T; ++J, ++blocks) {
        auto v = cover[{(int)k, I, J}];
        std::sort(v.begin(), v.end());
        int e = 0;
        for (const auto& r : v) {
          if (r.first != e) fail("stages not contiguous", n, m, C);
          e = r.second;
        }
        if (e != 4 * S) fail("stages not covered", n, m, C);
      }
  }
  if (cover.size() != blocks) fail("blocks", n, m, C);
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
  for (int64_t n : {1, 63, 64, 128, 129, 256, 257, 384, 385, 700, 1501, 4096, 5000, 9999, 20000})
    for (int64_t m : {1, 288, 289, 1000, 30011, 100000, 500000, 2097151})
      for (int c : {1, 5, 74, 76}) {
        check(ibs::sweep_plan(n, m, c), {{n, m}}, c);
        ++lists;
      }
  std::mt19937 g(1);
  for (int rep = 0; rep < 60; ++rep) {
    std::vector<std::pair<int64_t, int64_t>> shapes(1 + g() % 40);
    for (auto& s : shapes) s = {1 + g() % (rep % 3 ? 3000 : 300), 1 + g() % (rep % 5 ? 80000 : 2000)};
    for (int c : {5, 76}) {
      check(ibs::sweep_plan_batch(shapes, c), shapes, c);
      ++lists;
    }
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
