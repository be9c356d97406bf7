// Shared declarations of the libsdllm CUDA sources (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sdllm.h"

namespace sdllm {

constexpr int kMaxRows = 256;         // b * G rows of one KV head handled by one CTA
constexpr int kMaxSplits = 64;        // key-axis splits per (sequence, KV head)
// Workspace of the attention calls: [status word][counters][everything else]. One workspace serves calls of every kind in turn,
// and each call finds its counters at zero because the one before left them so; a call therefore keeps its data out of all of
// the first kWsDataOffset bytes, also when its own plan uses no counter.
constexpr size_t kWsStatusBytes = 256;
constexpr size_t kWsCounters = 192;   // the query-row kernel counts per (sequence, KV head, row tile) and splits the keys of at most half
                                      // as many of these as there are SMs (umma_tail_is_fused); the streaming kernel takes two
constexpr size_t kWsDataOffset = kWsStatusBytes + kWsCounters * sizeof(int32_t);
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// How one attention launch is cut into CTAs; a pure function of the description so that the workspace
// query and the launch always agree.
struct AttnPlan {
  int key_tile;     // keys per pipeline stage
  int m_warps;      // warps along the query rows (16 rows each, bf16) / row chunks (32 rows each, fp32)
  int c_warps;      // warps along the keys of a tile (bf16 only)
  int warp_keys;    // keys per warp per tile (cp.async bf16 kernel)
  int stages;       // shared-memory pipeline depth
  int cluster;      // > 1: the key splits of a unit form a thread-block cluster and merge through distributed shared memory
  int splits;       // partials per (sequence, KV head) left in the workspace (1 = final output written directly)
  int threads;
  size_t smem_bytes;
  int kind;         // 0: cp.async kernels (fp32 FMA / bf16 mma.sync); tcgen05 kernels - 2: attention pass of the probability saliency
                    // (attn_umma.cu), 3: keys on the accumulator rows (key splits merge inside their cluster), 4: queries on the
                    // accumulator rows, two softmax warpgroups (attn_pair.cu)
  int key_tile2;    // tcgen05 kernel: keys per tile of source 2
  int rep;          // tcgen05 kernel: replicas of the query rows along the 128 accumulator rows
  int row_tiles;    // tcgen05 kernel: 128-row tiles of the b*G rows
  bool fused_tail;  // nothing is left to launch_merge_pool: the attention launch merges the partials and pools the scores itself
  bool persistent;  // key-row kernel, streaming variant: one resident CTA per SM walks the units
  size_t part_rows; // partial rows per (sequence, KV head) in the workspace (0: none)
  int kv_share = 1; // key-row kernel, reuse step: units that the query rows of a KV head are shared out to
  size_t n_counters;// counters that the kernel uses, of the workspace's kWsCounters
};

// Key sources of one attention launch. The virtual key axis is [src1 rows 0..n1) ++ [src2 rows 0..n2).
// refresh: src1 = full K/V with n1 = seq_len[i], n2 = 0.  reuse: src1 = compacted cache with n1 = kept_cnt[i],
// src2 = the block's fresh rows with n2 = b.
struct AttnParams {
  const void* q;
  const void* k1; const void* v1;
  const void* k2; const void* v2;
  const int32_t* n1_per_seq;   // nullable -> n1_max
  const int32_t* block_off;    // refresh only
  void* out;                   // nullable
  float* lse;                  // nullable
  float* part_o;               // [B][Hkv][splits][M][D]
  float* part_ml;              // [B][Hkv][splits][M][2]  (running max in log2 units, running sum)
  float* raw_scores;           // [B][Hkv][n1_max] or null
  int B, Hq, Hkv, G, b, M;     // M = G * b rows per KV head
  int n1_max, n2;
  int splits;                  // partials per (sequence, KV head) in the workspace
  int splits_total;            // CTAs along the key axis per (sequence, KV head) = splits * cluster size
  int32_t* status;             // device status word: set non-zero when a bounded wait gave up
  long long wait_cycles;       // limit of an abortable device-side wait, in clock cycles
  int32_t* counters;           // completion counters (tcgen05 kernel), zero between calls
  float* pooled;               // refresh with a fused tail: pooled scores [B][Hkv][n1_max], else null
  int window, pool_kind, per_region;
  int releases_late;           // key-row kernel: the next launch may start once this one has seen everything before it complete, not earlier
  const float* lse_in;         // probability saliency, second pass: log-sum-exp of every block row [B][Hq][b]
  int unfolded;                // the key splits are folded, and the saliency is pooled, by the launch behind
  int want_scores;             // compute mean-query logit scores for src1 keys
  float scale;                 // softmax scale
  float scale_log2;            // scale * log2(e)
  int64_t q_stride[3], k1_stride[3], k2_stride[3], o_stride[3];
};

struct MergeParams {
  const float* part_o; const float* part_ml;
  void* out; float* lse;
  int B, Hq, Hkv, G, b, M, D, splits, dtype;
  int64_t o_stride[3];
  int merge_blocks;            // blocks [0, merge_blocks) merge; the rest pool
  // pooling of raw scores -> pooled scores
  const float* raw_scores; float* pooled;
  const int32_t* seq_len; const int32_t* block_off;
  int Lmax, window, pool_kind, per_region;
};

struct SelectParams {
  const float* pooled; const int32_t* seq_len; const int32_t* block_off;
  int32_t* kept_idx; int32_t* kept_cnt;
  int B, Hkv, Lmax, b, n_keep_max, mode;
  double retention;
  int gather_follows;          // selection alone: the next kernel in the stream is the gather, which waits for this one before it reads
  int early_inputs;            // fused kernel: seq_len and block_off are read ahead of the grid dependency
  // fused kernel, where it pools the saliency itself (raw: the unpooled saliency by absolute position, else null)
  const float* raw;
  float* pooled_out;
  int window, pool_kind;
};

// Fold of an attention call's key splits by the kernel behind it (partial rows as the attention kernels leave them).
struct FoldParams {
  const float* part_o; const float* part_ml;
  void* out; float* lse;
  int Hq, G, b, M, D, splits, dtype;
  int row_tiles;               // > 0: query-row kernel, [row tile][split][D / 4][128 rows]; 0: [split][M][D]
  int64_t o_stride[3];
  int ctas;                    // CTAs per (sequence, KV head) that fold; 0: nothing to fold
};

struct CompactParams {
  const void* k; const void* v; const int32_t* kept_idx; const int32_t* kept_cnt;
  void* k_c; void* v_c;
  int B, Hkv, n_keep_max, row_bytes, Lmax;
  int64_t kv_stride_bytes[3], c_stride_bytes[3];
};

struct AttnWorkspace {         // offsets in bytes; what lies at an offset ends where the next one begins
  size_t part_o, part_ml, raw, lse, total;
};
AttnWorkspace attn_workspace(const sdllm_desc* d, const AttnPlan& pl, bool scores);
// small: a reuse step of grouped heads takes the plan with the smaller workspace where there are two.
AttnPlan plan_attention(int dtype, int D, int M, int b, int B, int Hkv, int n1_max, int n2, bool prob_scores, bool small = false);
cudaError_t launch_prob_saliency(const AttnParams& p, int D, cudaStream_t st);    // second pass of the probability saliency

bool umma_tail_is_fused(const AttnPlan& pl, int D, int M);
bool umma_supported(int dtype, int D, int M, int b);
// Full-sequence attention (attn_dense.cu).
struct DenseCall {
  const void *q, *k, *v;
  const int64_t *q_stride, *kv_stride, *o_stride;
  const int32_t* seq_len;
  void* out; float* lse;
  void* workspace; size_t workspace_bytes;
  int B, Hq, Hkv, L, D;
  float scale;
};
cudaError_t launch_dense(const DenseCall& c, cudaStream_t st);
int dense_launches(int B, int Hq, int L, int D);             // kernel launches of one call
struct DenseWorkspace {
  size_t part_o, part_ml, total;
};
DenseWorkspace dense_workspace(int B, int Hq, int L, int D);
cudaError_t launch_attn_partial(const AttnParams& p, const AttnPlan& plan, int dtype, int D, cudaStream_t st);
cudaError_t launch_merge_pool(const MergeParams& p, cudaStream_t st);
cudaError_t launch_select_topk(const SelectParams& p, cudaStream_t st);
cudaError_t launch_compact(const CompactParams& p, cudaStream_t st);
cudaError_t launch_select_compact(const SelectParams& p, const CompactParams& cp, cudaStream_t st);
// The same for unpooled saliency (p.raw), with the fold of the attention call in front; only where select_compact_is_fused or
// select_is_clustered.
bool select_is_clustered(int B, int Hkv, int Lmax, int b, int n_keep_max);
cudaError_t launch_pool_select_compact(const SelectParams& p, const CompactParams& cp, const FoldParams& fold, cudaStream_t st);
constexpr int kMaxFusedWindow = 63;          // widest pooling window of a launch that pools and selects (its ends take shared memory)
// Saliency, pooling, selection and gather without the attention, in one launch beside the one in front (refresh_select.cu).
bool score_select_supported(int D, int M, int units, int cand);
AttnPlan plan_attention_kt_beside(int D, int M, int B, int Hkv, int n1_max);       // the attention beside it
cudaError_t launch_score_select(const AttnParams& p, const SelectParams& sp, const CompactParams& cp, int D, cudaStream_t st);
bool select_compact_is_fused(int B, int Hkv, int Lmax, int b, int n_keep_max);
int gather_ctas(int B, int Hkv, int n_keep_max, int folds);       // CTAs per head that copy rows there, beside `folds` that fold

__host__ __device__ inline int keep_count_total(int pre, int suf, double r, int mode, int* n_pre, int* n_suf) {
  // Algorithm 1: n = floor(|I| * r) in double; the other policies are described in sdllm.h.
  auto clampll = [](long long x, int hi) { return (int)(x < 0 ? 0 : (x > hi ? hi : x)); };
  if (mode == SDLLM_SELECT_JOINT_FLOOR) {
    *n_pre = -1; *n_suf = -1;
    return clampll((long long)floor((double)(pre + suf) * r), pre + suf);
  }
  if (mode == SDLLM_SELECT_PER_REGION_CEIL) {
    *n_pre = clampll((long long)ceil((double)pre * r), pre);
    *n_suf = clampll((long long)ceil((double)suf * r), suf);
    return *n_pre + *n_suf;
  }
  *n_pre = clampll((long long)floor((double)pre * r), pre);
  *n_suf = suf;
  return *n_pre + *n_suf;
}

}  // namespace sdllm
