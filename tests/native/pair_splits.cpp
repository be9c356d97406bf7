// Prints the key splits that the query-row kernel's planner takes for a refresh step, for every "query rows, units, key tiles" of
// the arguments.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "common.cuh"
#include "tuning.cuh"

namespace sdllm {
AttnPlan plan_attention_pair(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn);
}

int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3)
    printf("%d\n", sdllm::plan_attention_pair(128, atoi(argv[i]), 32, 1, atoi(argv[i + 1]), 128 * atoi(argv[i + 2]), 0, sdllm::Tuning{}).splits);
  return 0;
}
