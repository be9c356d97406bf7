// Walks the launch planners over shapes (no GPU needed) and checks that no attention call keeps data in the part of the workspace
// that holds the status word and the counters. Prints the first offender, or how many plans of each kind it saw.
#include <math.h>
#include <stdio.h>

#include "common.cuh"
#include "tuning.cuh"

namespace sdllm {
AttnPlan plan_attention_kt(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn);
AttnPlan plan_attention_pair(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn);
AttnPlan plan_attention_umma(int D, int M, int b, int B, int Hkv, int n1_max, const Tuning& tn);
}  // namespace sdllm
using namespace sdllm;

int main() {
  const size_t counters_end = kWsStatusBytes + kWsCounters * 4;
  long long counting = 0, streaming = 0, partial_rows = 0, dense_cut = 0;
  const int batches[] = {1, 2, 4, 10, 16, 64}, groups[] = {1, 2, 4, 7, 8}, blocks[] = {8, 16, 32, 64, 128};
  const int kv_heads[] = {1, 2, 4, 8, 32, 80, 96}, lengths[] = {160, 704, 768, 864, 1280, 2048, 4352, 32768};
  for (int B : batches) for (int Hkv : kv_heads) for (int L : lengths) for (int D : {64, 128}) {
    for (int G : groups) for (int b : blocks) for (int splits : {0, 3}) for (bool refresh : {true, false}) for (bool prob : {false, true}) {
      const int M = G * b;
      if (M > 256 || (prob && !refresh)) continue;
      sdllm_desc d{};
      d.struct_size = sizeof(d); d.batch = B; d.n_q_heads = G * Hkv; d.n_kv_heads = Hkv; d.head_dim = D; d.seq_len_max = L; d.block_len = b;
      d.dtype = SDLLM_BF16; d.score = prob ? SDLLM_SCORE_PROB_MEAN : SDLLM_SCORE_LOGIT_MEAN; d.n_keep_max = (int)(0.9 * (L - b));
      Tuning tn;
      tn.splits = splits;
      const int n1 = refresh ? L : d.n_keep_max, n2 = refresh ? 0 : b;
      for (int kind = 0; kind < 4; ++kind) {
        if (kind == 1 && (M > 128 || M % 4 != 0)) continue;
        if (kind == 3 && (!prob || b % 16 != 0 || (M > 128 && 128 % b != 0))) continue;
        const AttnPlan pl = kind == 0   ? plan_attention(SDLLM_F32, D, M, b, B, Hkv, n1, n2, false)
                            : kind == 1 ? plan_attention_kt(D, M, b, B, Hkv, n1, n2, tn)
                            : kind == 2 ? plan_attention_pair(D, M, b, B, Hkv, n1, n2, tn)
                                        : plan_attention_umma(D, M, b, B, Hkv, n1, tn);
        const AttnWorkspace w = attn_workspace(&d, pl, refresh);
        const bool counts = pl.persistent || (pl.kind == 2 && pl.splits > 1 && umma_tail_is_fused(pl, D, M));
        const size_t rows = (size_t)B * Hkv * pl.part_rows;
        if (w.part_o < counters_end || w.part_ml < w.part_o + rows * D * 4 || w.raw < w.part_ml + rows * 8 ||
            w.lse < w.raw + (refresh ? (size_t)B * Hkv * L * 4 : 0) || w.total < w.lse + (prob ? (size_t)B * Hkv * M * 4 : 0) ||
            (counts && pl.n_counters > kWsCounters)) {
          printf("kind %d B %d Hkv %d G %d b %d D %d L %d refresh %d prob %d: counters %zu, data at %zu\n", kind, B, Hkv, G, b, D, L, refresh, prob,
                 pl.n_counters, w.part_o);
          return 1;
        }
        counting += counts && !pl.persistent; streaming += pl.persistent; partial_rows += pl.part_rows > 0;
      }
    }
    const DenseWorkspace w = dense_workspace(B, Hkv, L, D);
    const size_t rows = (w.part_ml - w.part_o) / D / 4;
    if (w.total != kWsStatusBytes && (w.part_o < counters_end || w.total < w.part_ml + rows * 8)) {
      printf("dense B %d Hq %d L %d D %d: data at %zu\n", B, Hkv, L, D, w.part_o);
      return 1;
    }
    dense_cut += rows > 0;
  }
  printf("%lld %lld %lld %lld\n", counting, streaming, partial_rows, dense_cut);
  return 0;
}
