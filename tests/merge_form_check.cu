// Host-side check of the merge Gram's choice between reading its rows where they lie
// and reading a permuted copy. For each shape given on the command line (B N_v keep D
// SMs) prints the halves of the chosen plan's groups and "direct" or "copy"; after a
// first argument "search", compares the plans of both group sizes with those of a search
// that deals every tile of every candidate, and prints "ok" with the host time of a shape
// not seen before over that of one such search (512-row groups read from the copy). Host
// code only.
#include "../paper_2608_25332_gb300/csrc/merge_pair_tc.cu"

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cstring>

namespace provip {
int make_tmap_bf16_2d(CUtensorMap*, const void*, uint64_t, uint64_t, uint64_t, uint32_t) { return -1; }
}  // namespace provip

using namespace provip;

// the split whose busiest pair has the fewest clocks, every candidate's tiles dealt one by
// one as the kernel deals them
static bool search(int halves, bool direct, int B, int n_pruned, int keep, int D, int sms, MergePairPlan* p) {
  const int n_quads = (n_pruned + halves * 256 - 1) / (halves * 256), n_k = (D + 63) / 64;
  const double pace = (double)(direct ? kDirectPace : kBoxPace)[halves - 1];
  const long long Q = (long long)B * n_quads;
  bool found = false;
  auto consider = [&](int n_lo, long long x_hi) {
    MergePairPlan c = {};
    c.halves = halves;
    c.direct = direct;
    c.n_quads = n_quads;
    c.Q = (int)Q;
    c.n_lo = n_lo;
    c.x_hi = (int)x_hi;
    c.n_slots = n_lo + (x_hi > 0);
    if (c.n_slots > kMergeMaxSplit) return;
    c.T = (int)(Q * n_lo + x_hi);
    c.P = std::min(c.T, sms / 2);
    std::vector<double> load(c.P, 0.0);
    for (int pr = 0; pr < c.P; ++pr)
      for (int r = 0, k; (k = pair_deal_tile(c, pr, r)) >= 0; ++r) {
        const PairTile g = pair_tile(c, n_pruned, keep, k);
        if (g.nv < 1 || g.nv > 256) return;
        int j = 0;
        while (j < c.n_heights && c.heights[j] != g.N / 2) ++j;
        if (j == c.n_heights) {
          if (j == kMergePairHeights) return;
          c.heights[c.n_heights++] = g.N / 2;
        }
        load[pr] += n_k * fmax((g.has1 ? 4.0 : 2.0) * g.N, pace) + 9000.0;
      }
    c.clocks = *std::max_element(load.begin(), load.end()) +
               (direct ? 0.0 : kCopyClocksPerByte * 4.0 * B * (n_pruned + keep) * (double)D);
    if (!found || c.clocks < p->clocks) *p = c;
    found = true;
  };
  for (int n_lo = (keep + 255) / 256; n_lo <= kMergeMaxSplit; ++n_lo)
    for (int m = 0; m <= 4; ++m) {
      const long long x_hi = m == 0 ? 0 : (long long)m * (sms / 2) - Q * n_lo;
      if (m == 0 || (x_hi > 0 && x_hi < Q)) consider(n_lo, x_hi);
    }
  return found;
}

static double micros(std::chrono::steady_clock::time_point t) {
  return std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t).count();
}

static int check_search(int B, int N_v, int keep, int D, int sms) {
  const int n_pruned = N_v - keep;
  for (int halves = 1; halves <= 2; ++halves) {
    MergePairPlan p, copy, want;
    const bool has = halves == 1 ? merge_pair_half_plan(B, n_pruned, keep, D, sms, &p)
                                 : merge_pair_plan(B, n_pruned, keep, D, sms, &p);
    const bool has_copy = search(halves, false, B, n_pruned, keep, D, sms, &copy);
    const bool has_direct = search(halves, true, B, n_pruned, keep, D, sms, &want);
    if (has_copy && (!has_direct || want.clocks >= copy.clocks)) want = copy;
    if (has != (has_copy || has_direct)) return printf("B=%d N_v=%d keep=%d D=%d: found %d\n", B, N_v, keep, D, has), 1;
    if (has && (p.halves != halves || p.direct != want.direct || p.n_quads != want.n_quads || p.Q != want.Q ||
                p.n_lo != want.n_lo || p.x_hi != want.x_hi || p.T != want.T || p.P != want.P ||
                p.n_slots != want.n_slots || p.clocks != want.clocks))
      return printf("B=%d N_v=%d keep=%d D=%d halves=%d: %d + %d ranges, %s, %.1f clocks; best %d + %d, %s, %.1f\n", B,
                    N_v, keep, D, halves, p.n_lo, p.x_hi, p.direct ? "direct" : "copy", p.clocks, want.n_lo, want.x_hi,
                    want.direct ? "direct" : "copy", want.clocks), 1;
  }
  // the quickest of 16 shapes not seen before that take the same plans
  double miss = 1e30, one = 1e30;
  const int n_k = (D + 63) / 64;
  for (int i = 0; i < 16; ++i) {
    MergePairPlan p;
    auto t = std::chrono::steady_clock::now();
    merge_pair_best(B, n_pruned, keep, n_k * 64 + 64 * (i + 1), sms, &p);
    miss = std::min(miss, micros(t));
    t = std::chrono::steady_clock::now();
    search(2, false, B, n_pruned, keep, n_k * 64 + 64 * (i + 1), sms, &p);
    one = std::min(one, micros(t));
  }
  return printf("ok %.3f (%.1f us, one %.1f us)\n", miss / one, miss, one), 0;
}

int main(int argc, char** argv) {
  const bool s = argc > 1 && strcmp(argv[1], "search") == 0;
  for (int i = s ? 2 : 1; i + 4 < argc; i += 5) {
    const int B = atoi(argv[i]), N_v = atoi(argv[i + 1]), keep = atoi(argv[i + 2]), D = atoi(argv[i + 3]),
              sms = atoi(argv[i + 4]);
    if (s) {
      if (check_search(B, N_v, keep, D, sms)) return 1;
      continue;
    }
    MergePairPlan p;
    if (!merge_pair_best(B, N_v - keep, keep, D, sms, &p)) return printf("noplan\n"), 1;
    printf("%d %s\n", p.halves, p.direct ? "direct" : "copy");
  }
}
