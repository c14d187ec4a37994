// Host-side check of the merge Gram's tile plan with 256-row groups on SM pairs and
// of the choice between it and 512-row groups: for each shape given on the command
// line (B N_v keep D SMs), every pruned row of every sample must get each partial
// slot written exactly once, no tile may use a second half, every range must be
// 1..256 columns wide with a planned box height, every tile dealt to one pair; and
// the chosen form must be the one with the fewer clocks. Prints "ok" and the chosen
// form per shape or the first violation. Host code only.
#include "../paper_2608_25332_gb300/csrc/merge_pair_tc.cu"

#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>

namespace provip {
int make_tmap_bf16_2d(CUtensorMap*, const void*, uint64_t, uint64_t, uint64_t, uint32_t) { return -1; }
}  // namespace provip

using namespace provip;

static int check(int B, int N_v, int keep, int D, int sms) {
  const int n_pruned = N_v - keep;
  MergePairPlan p, two, best;
  const bool has1 = merge_pair_half_plan(B, n_pruned, keep, D, sms, &p);
  const bool has2 = merge_pair_plan(B, n_pruned, keep, D, sms, &two);
  const bool has = merge_pair_best(B, n_pruned, keep, D, sms, &best);
  if (has != (has1 || has2) || (has1 && p.halves != 1) || (has2 && two.halves != 2)) return printf("forms\n"), 1;
  if (has) {
    const int want = has1 && (!has2 || p.clocks < two.clocks) ? 1 : 2;
    if (best.halves != want) return printf("B=%d N_v=%d keep=%d: form %d\n", B, N_v, keep, best.halves), 1;
  }
  if (!has1) return printf("noplan\n"), 0;
  if (p.P < 1 || p.P > sms / 2 || p.n_slots < 1 || p.n_slots > kMergeMaxSplit) return printf("bad plan\n"), 1;
  std::vector<unsigned char> cover((size_t)B * n_pruned * p.n_slots, 0);
  std::set<int> seen;
  for (int pair = 0; pair < p.P; ++pair)
    for (int r = 0, k; (k = pair_deal_tile(p, pair, r)) >= 0; ++r) {
      if (!seen.insert(k).second || k >= p.T) return printf("tile %d dealt twice or out of range\n", k), 1;
      const PairTile g = pair_tile(p, n_pruned, keep, k);
      bool h_ok = false;
      for (int j = 0; j < p.n_heights; ++j) h_ok |= p.heights[j] == g.N / 2;
      if (g.has1 || g.nv < 1 || g.nv > 256 || g.N % 32 || g.N < g.nv || !h_ok || g.c0 + g.nv > keep || g.b >= B)
        return printf("tile %d\n", k), 1;
      const bool spare = g.t + 1 == g.n && g.n < p.n_slots;
      for (int pos = g.m0; pos < g.m0 + 256 && pos < n_pruned; ++pos)
        for (int sl = g.t; sl <= (spare ? g.t + 1 : g.t); ++sl) ++cover[((size_t)g.b * n_pruned + pos) * p.n_slots + sl];
    }
  if ((int)seen.size() != p.T) return printf("%zu of %d tiles dealt\n", seen.size(), p.T), 1;
  for (size_t i = 0; i < cover.size(); ++i)
    if (cover[i] != 1) return printf("B=%d N_v=%d keep=%d: written %d times\n", B, N_v, keep, cover[i]), 1;
  printf("ok %d\n", best.halves);
  return 0;
}

int main(int argc, char** argv) {
  int rc = 0;
  for (int i = 1; i + 4 < argc; i += 5)
    rc |= check(atoi(argv[i]), atoi(argv[i + 1]), atoi(argv[i + 2]), atoi(argv[i + 3]), atoi(argv[i + 4]));
  return rc;
}
