// Prints the launches of a dense step of one sequence, for every "head dimension, query heads, length" of the arguments: 1 with all units whole,
// 2 with the cut units in front (or all units cut), 3 with the cut units behind the whole ones.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "common.cuh"

int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3) printf("%d\n", sdllm::dense_launches(1, atoi(argv[i + 1]), atoi(argv[i + 2]), atoi(argv[i])));
  return 0;
}
