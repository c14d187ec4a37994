// Host-side check of the merge Gram's choice between reading its rows where they lie
// and reading a permuted copy: for each shape given on the command line (B N_v keep D
// SMs) prints the halves of the chosen plan's groups and "direct" or "copy". Host
// code only.
#include "../paper_2608_25332_gb300/csrc/merge_pair_tc.cu"

#include <cstdio>
#include <cstdlib>

namespace provip {
int make_tmap_bf16_2d(CUtensorMap*, const void*, uint64_t, uint64_t, uint64_t, uint32_t) { return -1; }
}  // namespace provip

int main(int argc, char** argv) {
  for (int i = 1; i + 4 < argc; i += 5) {
    const int N_v = atoi(argv[i + 1]), keep = atoi(argv[i + 2]);
    provip::MergePairPlan p;
    if (!provip::merge_pair_best(atoi(argv[i]), N_v - keep, keep, atoi(argv[i + 3]), atoi(argv[i + 4]), &p))
      return printf("noplan\n"), 1;
    printf("%d %s\n", p.halves, p.direct ? "direct" : "copy");
  }
}
