// Host-side check of where the critical text rows come first on the stream of the
// pre-LLM pass: for each shape given on the command line (B N_v N_t D SMs) prints 1 or 0.
// Host code only.
#include "../paper_2608_25332_gb300/csrc/similarity_tc.cu"

#include <cstdio>
#include <cstdlib>

namespace provip {
int make_tmap_bf16_2d(CUtensorMap*, const void*, uint64_t, uint64_t, uint64_t, uint32_t) { return -1; }
bool merge_pair_usable(const SimArgs&) { return false; }
bool merge_pair_best(int, int, int, int, int, MergePairPlan*) { return false; }
cudaError_t merge_argmax_pair_launch(const SimArgs&, const int*, int, const float*, const int*, const void*,
                                     const MergePairPlan&, float*, int*, cudaStream_t) {
  return cudaErrorNotSupported;
}
}  // namespace provip

int main(int argc, char** argv) {
  for (int i = 1; i + 4 < argc; i += 5) {
    provip::SimArgs a = {};
    a.B = atoi(argv[i]);
    a.N_v = atoi(argv[i + 1]);
    a.N_t_max = atoi(argv[i + 2]);
    a.D = atoi(argv[i + 3]);
    a.dtype = 1;
    printf("%d\n", provip::crit_leads(a, atoi(argv[i + 4])) ? 1 : 0);
  }
}
