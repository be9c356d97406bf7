// Prints how many units the planner shares out a KV head's query rows to in a reuse step (0: none), for every "head dimension, query heads
// per KV head, block length, KV heads, cached keys" of the arguments.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "common.cuh"
#include "tuning.cuh"

namespace sdllm {
bool plan_attention_units(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn, bool small, AttnPlan* pl);
}

int main(int argc, char** argv) {
  for (int i = 1; i + 4 < argc; i += 5) {
    int a[5];
    for (int j = 0; j < 5; ++j) a[j] = atoi(argv[i + j]);
    sdllm::AttnPlan pl{};
    printf("%d\n", sdllm::plan_attention_units(a[0], a[1] * a[2], a[2], 1, a[3], a[4], a[2], sdllm::Tuning{}, false, &pl) ? pl.kv_share : 0);
  }
  return 0;
}
