// Largest relative errors of poly_exp2 and of fast_exp2 against exp2 in 64 bits, over evenly spaced arguments of [-126, 8] and over
// ones of every exponent, and what poly_exp2 makes of arguments that are not finite.
#include <cuda.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "common.cuh"

namespace {
#include "umma_ptx.cuh"

constexpr int kBlocks = 1024, kThreads = 256, kPerThread = 64;

__global__ void errors(unsigned* worst) {
  for (int i = 0; i < kPerThread; ++i) {
    const unsigned n = (blockIdx.x * kPerThread + i) * kThreads + threadIdx.x;
    // evenly spaced, and any mantissa with an exponent of 2^-30 to 2^6
    const float even = -126.f + 134.f * (float)n / (float)(kBlocks * kThreads * kPerThread);
    const float spread = -__uint_as_float(((97u + n % 37u) << 23) | (n * 2654435761u >> 9));
    const float x[2] = {even, fmaxf(spread, -126.f)};
    float y[2];
    poly_exp2(x[0], x[1], y[0], y[1]);
    for (int k = 0; k < 2; ++k) {
      const double want = exp2((double)x[k]);
      atomicMax(worst + k, __float_as_uint((float)fabs((double)y[k] / want - 1.0)));
      if (x[k] > -125.f) atomicMax(worst + 2, __float_as_uint((float)fabs((double)fast_exp2(x[k]) / want - 1.0)));   // (it flushes below 2^-126)
    }
  }
}
__global__ void specials(float* out) {
  poly_exp2(NAN, -INFINITY, out[0], out[1]);
  poly_exp2(-1e30f, -126.5f, out[2], out[3]);
  poly_exp2(0.f, 8.f, out[4], out[5]);
  out[6] = kNanSum;
}
}  // namespace

int main() {
  unsigned* worst;
  float *out, e[3], s[7];
  if (cudaMallocManaged(&worst, 3 * sizeof(unsigned)) != cudaSuccess || cudaMallocManaged(&out, 7 * sizeof(float)) != cudaSuccess) return 2;
  for (int i = 0; i < 3; ++i) worst[i] = 0;
  errors<<<kBlocks, kThreads>>>(worst);
  specials<<<1, 1>>>(out);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  memcpy(e, worst, sizeof(e));
  memcpy(s, out, sizeof(s));
  printf("%.3e %.3e %.3e\n", e[0], e[1], e[2]);
  for (float x : s) printf("%.9e ", x);
  printf("\n");
  return 0;
}
