// Top-k selection over the pooled importance scores and the K/V gather-compaction
// (Algorithm 1: "n <- floor(|I| r)", "TopKIndices(I, n)", "Select(K_f, I)", "Select(V_f, I)").
#include <cuda.h>

#include <type_traits>

#include "common.cuh"
#include "fold.cuh"
#include "tuning.cuh"

namespace sdllm {
namespace {

#include "select_common.cuh"

// The fold's parameters travel only with the launches that fold (RAW).
struct NoFold {};
template <bool RAW>
using FoldOf = std::conditional_t<RAW, FoldParams, NoFold>;

// Selection alone: CS CTAs of SW warps per (sequence, KV head).
// RAW (clusters): the scores are the attention kernel's unpooled saliency; every CTA brings its slice of them and half a window either
// side into shared memory, pools it into its keys and writes its pooled scores, and a second cluster per head folds the attention's
// key splits (see select_gather_kernel; 8 heads x 32736 candidates: the refresh without the launch in between 79.1 -> 74.4 us).
template <int SW, int KPT, int CS, bool RAW>
__global__ void __launch_bounds__(32 * SW) select_topk_kernel(const SelectParams p, const FoldOf<RAW> fold) {
  __shared__ __align__(16) SelectShared<SW, CS> sh;
  constexpr int NT = 32 * SW;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = CS > 1 ? (int)cluster_rank() : 0;
  const int g = blockIdx.y, bi = blockIdx.z;
  if constexpr (RAW) {
    if (blockIdx.x >= CS) {                            // (a whole cluster)
      asm volatile("griddepcontrol.wait;\n" ::: "memory");
      if (p.gather_follows) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
      fold_head<NT>(fold, bi * p.Hkv + g, bi, g, rank);
      return;
    }
  }
  sh.clear(tid, NT);
  if constexpr (CS > 1) {
    cluster_barrier();                                 // every peer runs and has cleared its histograms
  } else {
    __syncthreads();
  }
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (p.gather_follows) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const HeadPlace h = place_head(p, p.seq_len ? p.seq_len[bi] : p.Lmax, p.block_off[bi]);
  const int slice = (h.C + CS - 1) / CS;
  const int s_lo = min(rank * slice, h.C), s_hi = min(s_lo + slice, h.C);
  const int kpt = min((s_hi - s_lo + NT - 1) / NT, KPT);
  const int c0 = s_lo + warp * 32 * kpt + lane;
  const int64_t head_row = (int64_t)(bi * p.Hkv + g) * p.Lmax;
  uint32_t key[KPT];
  if constexpr (RAW) {
    extern __shared__ float raw_s[];                   // candidates s_lo - w up to s_hi + w
    const int w = (p.window - 1) / 2, first = s_lo - w;
    for (int i = tid; i < s_hi - s_lo + 2 * w; i += NT) {
      const int c = first + i;
      if (c >= 0 && c < h.C) raw_s[i] = __ldcg(p.raw + head_row + (c < h.o ? c : c + h.b));
    }
    __syncthreads();
    const bool per_region = p.mode != SDLLM_SELECT_JOINT_FLOOR;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const int c = c0 + 32 * j;
      key[j] = 0u;
      if (j < kpt && c < s_hi) {
        const int lo = max(per_region && c >= h.o ? h.o : 0, c - w), hi = min(per_region && c < h.o ? h.o : h.C, c + w + 1);
        float mx = -INFINITY, sum = 0.f;
        for (int t = lo; t < hi; ++t) {
          mx = fmaxf(mx, raw_s[t - first]);
          sum += raw_s[t - first];
        }
        const float x = p.pool_kind == SDLLM_POOL_MAX ? mx : sum / (float)p.window;
        p.pooled_out[head_row + (c < h.o ? c : c + h.b)] = x;
        key[j] = score_key(x);
      }
    }
    for (int pos = rank * NT + tid; pos < p.Lmax; pos += CS * NT)       // the block's own positions and the padding
      if (pos >= h.C + h.b || (pos >= h.o && pos < h.o + h.b)) p.pooled_out[head_row + pos] = -INFINITY;
  } else {
    load_keys(key, p.pooled + head_row, h, kpt, c0, s_hi);
  }
  int32_t* out = p.kept_idx + (int64_t)(bi * p.Hkv + g) * p.n_keep_max;
  for (int i = h.kept + rank * NT + tid; i < p.n_keep_max; i += CS * NT) out[i] = -1;
  if (g == 0 && rank == 0 && tid == 0) p.kept_cnt[bi] = h.kept;
  select_head<SW, KPT, CS>(h, key, c0, sh, rank, [&](int w, int c) { out[w] = c < h.o ? c : c + h.b; });
  if constexpr (CS > 1) cluster_barrier();             // nobody leaves while a peer may still write to its shared memory
}

// More candidates than the registers of a cluster (or, on request, of a CTA) hold: one CTA per head reads the scores from
// global memory in every pass.
constexpr int SELG_THREADS = 1024;
__global__ void __launch_bounds__(SELG_THREADS) select_topk_global_kernel(const SelectParams p) {
  constexpr int NW = SELG_THREADS / 32;
  __shared__ uint32_t hist[256];
  __shared__ uint32_t warp_tot[2][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = blockIdx.x, bi = blockIdx.y;
  const HeadPlace h = place_head(p, p.seq_len ? p.seq_len[bi] : p.Lmax, p.block_off[bi]);
  const float* sc = p.pooled + (int64_t)(bi * p.Hkv + g) * p.Lmax;
  int32_t* out = p.kept_idx + (int64_t)(bi * p.Hkv + g) * p.n_keep_max;
  auto cand_pos = [&](int c) { return c < h.o ? c : c + h.b; };
  auto key_at = [&](int c) -> uint32_t { return score_key(sc[cand_pos(c)]); };
  uint32_t run_out = 0;
#pragma unroll 1
  for (int si = 0; si < 2; ++si) {
    const int c_lo = si == 0 ? 0 : h.c1, c_hi = si == 0 ? h.c1 : h.C, n = si == 0 ? h.n0 : h.n1;
    if (n <= 0 || c_hi <= c_lo) continue;
    uint32_t thr = 0u, need_eq = 0u;
    const bool take_all = n >= c_hi - c_lo;
    if (!take_all) {
      uint32_t remaining = (uint32_t)n;
      for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const uint32_t himask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
        __syncthreads();
        if (tid < 256) hist[tid] = 0u;
        __syncthreads();
        for (int c = c_lo + tid; c < c_hi; c += SELG_THREADS) {
          const uint32_t k = key_at(c);
          if ((k & himask) == thr) atomicAdd(&hist[(k >> shift) & 0xFFu], 1u);
        }
        __syncthreads();
        uint32_t bin = 255u;                           // (every thread walks the bins from the top: a handful of them)
        while (hist[bin] < remaining) remaining -= hist[bin--];
        thr |= bin << shift;
      }
      need_eq = remaining;
    }
    // ordered emission in rounds of one candidate per thread
    uint32_t gt_before = 0, eq_before = 0;
    const uint32_t below = (1u << lane) - 1u;
    for (int c_0 = c_lo; c_0 < c_hi; c_0 += SELG_THREADS) {
      const int c = c_0 + tid;
      const uint32_t k = c < c_hi ? key_at(c) : 0u;
      const bool gt = c < c_hi && (take_all || k > thr), eq = c < c_hi && !take_all && k == thr;
      const uint32_t m_gt = __ballot_sync(0xffffffffu, gt), m_eq = __ballot_sync(0xffffffffu, eq);
      __syncthreads();
      if (lane == 0) { warp_tot[0][warp] = __popc(m_gt); warp_tot[1][warp] = __popc(m_eq); }
      __syncthreads();
      const uint32_t tg = warp_tot[0][lane], te = warp_tot[1][lane];
      const uint32_t g0 = gt_before + __reduce_add_sync(0xffffffffu, lane < warp ? tg : 0u) + __popc(m_gt & below);
      const uint32_t e0 = eq_before + __reduce_add_sync(0xffffffffu, lane < warp ? te : 0u) + __popc(m_eq & below);
      if (gt || (eq && e0 < need_eq)) out[run_out + g0 + min(e0, need_eq)] = cand_pos(c);
      gt_before += __reduce_add_sync(0xffffffffu, tg);
      eq_before += __reduce_add_sync(0xffffffffu, te);
    }
    run_out += (uint32_t)n;
  }
  for (int i = h.kept + tid; i < p.n_keep_max; i += SELG_THREADS) out[i] = -1;
  if (g == 0 && tid == 0) p.kept_cnt[bi] = h.kept;
}

// ---------------------------------------------------------------------------------------------------------
// Gather: 16 bytes per thread, several rows of K and of V in flight per thread. Bound by HBM (rows read and written, zero rows
// written). The kernel of its own has many CTAs and takes two rows per thread: 512 heads of 2160 rows, 0.93 GB, 160 us with four,
// 148 with two, 185 with one; 190 with K and V in CTAs of their own. The fused kernel below has one CTA per SM and takes four.
constexpr int CP_ROWS_PER_THREAD = 4;
constexpr int CP_ROWS_ALONE = 2;

__global__ void __launch_bounds__(256) compact_kv_kernel(const CompactParams p) {
  const int lg = 31 - __clz(p.row_bytes / 16);         // log2 of the threads per row
  const int rows_per_pass = 256 >> lg;
  const int tid = threadIdx.x;
  const int c = tid & ((1 << lg) - 1);
  const int g = blockIdx.y, bi = blockIdx.z;
  const int32_t* idx = p.kept_idx + (int64_t)(bi * p.Hkv + g) * p.n_keep_max;
  const GatherHead h = gather_head(p, bi, g);
  const int row0 = blockIdx.x * rows_per_pass * CP_ROWS_ALONE + (tid >> lg);
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int cnt = min(max(__ldcg(p.kept_cnt + bi), 0), p.n_keep_max);

  uint4 kv[CP_ROWS_ALONE], vv[CP_ROWS_ALONE];
#pragma unroll
  for (int u = 0; u < CP_ROWS_ALONE; ++u) {
    const int i = row0 + u * rows_per_pass;
    kv[u] = make_uint4(0u, 0u, 0u, 0u);
    vv[u] = make_uint4(0u, 0u, 0u, 0u);
    if (i < cnt) {
      const int src = __ldcg(idx + i);
      if (src >= 0 && src < p.Lmax) {
        kv[u] = __ldg(reinterpret_cast<const uint4*>(h.k + (int64_t)src * p.kv_stride_bytes[2]) + c);
        vv[u] = __ldg(reinterpret_cast<const uint4*>(h.v + (int64_t)src * p.kv_stride_bytes[2]) + c);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < CP_ROWS_ALONE; ++u) {
    const int i = row0 + u * rows_per_pass;
    if (i < p.n_keep_max) {
      reinterpret_cast<uint4*>(h.k_c + (int64_t)i * p.c_stride_bytes[2])[c] = kv[u];
      reinterpret_cast<uint4*>(h.v_c + (int64_t)i * p.c_stride_bytes[2])[c] = vv[u];
    }
  }
}

// ---------------------------------------------------------------------------------------------------------
// Selection and gather in one launch (Algorithm 1 from "n <- floor(|I| r)" to the cache store), for batches of fewer heads
// than SMs. R CTAs share a (sequence, KV head): every one of them runs the whole selection of the head on its own - repeating
// it costs no time and needs no exchange - and keeps the positions of the r-th share of the (padded) list, which it writes
// to kept_idx and whose K and V rows it copies into the compacted cache (zero rows and -1 past the count). How many entries
// are kept is known beforehand, so the warps that do not select write the empty rows meanwhile; all warps copy.
// (With more heads than SMs the selections of one CTA after another stand still in front of the gathers, and a CTA per head
// is too coarse for a ragged batch: there the selection runs alone, in one wave, and the fine-grained gather behind it. A
// refresh of 16 sequences of 921 to 4352 tokens, 512 heads: 367 -> 344 us.)
//
// RAW: the scores are the attention kernel's unpooled saliency. Every CTA of a head brings the head's raw scores into shared
// memory, pools its candidates on the way into their keys (Algorithm 1, MaxPool1D(A, kernel_size = s, padding = s/2) over the
// candidate axis, the window cut off at the ends of the axis or, per region, of the region) and writes its share of the pooled
// scores; fold.ctas more CTAs per head fold the attention's key splits meanwhile. The launch that pooled and folded between the
// two, 3 to 4 us of a refresh, is gone (2 fp32 heads x 256 keys 13.7 -> 10.1 us, 28 / 4 heads x 4096 25.1 -> 22.0), and the
// key-row kernel ends with its merge (32 heads x 1280: 20.6 -> 20.1).
template <int SW, int KPT, bool RAW>
__global__ void __launch_bounds__(1024) select_gather_kernel(const SelectParams p, const CompactParams cp, const FoldOf<RAW> fold) {
  constexpr int NT = 1024;
  extern __shared__ int32_t kept_s[];                  // kept positions of this CTA's share of the list, then (RAW) the raw scores
  __shared__ __align__(16) SelectShared<SW, 1> sh;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x, g = blockIdx.y, bi = blockIdx.z;
  int R = gridDim.x;
  if constexpr (RAW) {
    R -= fold.ctas;
    if (r >= R) {
      asm volatile("griddepcontrol.wait;\n" ::: "memory");
      fold_head<NT>(fold, bi * p.Hkv + g, bi, g, r - R);
      return;
    }
  }
  for (int i = tid; i < (int)(sizeof(sh.hist) / 4); i += NT) (&sh.hist[0][0][0])[i] = 0u;
  // Ahead of the grid dependency: all that does not depend on the scores of the kernel in front (the caller's lengths and
  // block offsets are older than those).
  if (!p.early_inputs) asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const HeadPlace h = place_head(p, p.seq_len ? __ldcg(p.seq_len + bi) : p.Lmax, __ldcg(p.block_off + bi));
  const int kpt = min((h.C + 32 * SW - 1) / (32 * SW), KPT);
  const int c0 = warp * 32 * kpt + lane;
  const float* scores = (RAW ? p.raw : p.pooled) + (int64_t)(bi * p.Hkv + g) * p.Lmax;
  int32_t* out = p.kept_idx + (int64_t)(bi * p.Hkv + g) * p.n_keep_max;
  // this CTA's share: the kept entries [i_lo, i_hi) and the empty ones [z_lo, z_hi) of the head's list (R <= 16)
  const int pad = p.n_keep_max - h.kept;
  const int i_lo = r * h.kept / R, i_hi = (r + 1) * h.kept / R;
  const int z_lo = h.kept + r * pad / R, z_hi = h.kept + (r + 1) * pad / R;
  const int lg = 31 - __clz(cp.row_bytes / 16);        // log2 of the threads per row
  const GatherHead gh = gather_head(cp, bi, g);
  [[maybe_unused]] float* raw_s = RAW ? reinterpret_cast<float*>(kept_s + (p.n_keep_max + R - 1) / R + 1) : nullptr;
  __syncthreads();
  if (p.early_inputs) asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if constexpr (RAW) {
    const RawAxis axis(p, h);
    axis.clear_ends(raw_s, h.C, tid, NT);
    for (int c = tid; c < h.C; c += NT) raw_s[axis.at(c)] = __ldcg(scores + (c < h.o ? c : c + h.b));
    __syncthreads();
  }

  if (warp < SW) {
    uint32_t key[KPT];
    if constexpr (RAW) {
      pool_keys(key, RawAxis(p, h), raw_s, h.C, kpt, c0);
    } else {
      load_keys(key, scores, h, kpt, c0, h.C);
    }
    select_head<SW, KPT, 1>(h, key, c0, sh, 0, [&](int w, int c) {
      if (w >= i_lo && w < i_hi) kept_s[w - i_lo] = c < h.o ? c : c + h.b;
    });
  } else {
    const int t = tid - 32 * SW, nt = NT - 32 * SW;
    if (g == 0 && r == 0 && t == 0) p.kept_cnt[bi] = h.kept;
    if constexpr (RAW) write_pooled(p, raw_s, h, bi * p.Hkv + g, r, R, t, nt);
    write_empty_entries(cp, gh, out, z_lo, z_hi, t, nt);
  }
  __syncthreads();

  for (int i = i_lo + tid; i < i_hi; i += NT) out[i] = kept_s[i - i_lo];
  const int rows_per_pass = NT >> lg, c16 = tid & ((1 << lg) - 1);
#pragma unroll 1
  for (int i0 = i_lo + (tid >> lg); i0 < i_hi; i0 += CP_ROWS_PER_THREAD * rows_per_pass) {
    uint4 kv[CP_ROWS_PER_THREAD], vv[CP_ROWS_PER_THREAD];
#pragma unroll
    for (int u = 0; u < CP_ROWS_PER_THREAD; ++u) {
      const int i = i0 + u * rows_per_pass;
      if (i < i_hi) {
        const int64_t at = (int64_t)kept_s[i - i_lo] * cp.kv_stride_bytes[2];
        kv[u] = __ldg(reinterpret_cast<const uint4*>(gh.k + at) + c16);
        vv[u] = __ldg(reinterpret_cast<const uint4*>(gh.v + at) + c16);
      }
    }
#pragma unroll
    for (int u = 0; u < CP_ROWS_PER_THREAD; ++u) {
      const int i = i0 + u * rows_per_pass;
      if (i < i_hi) {
        reinterpret_cast<uint4*>(gh.k_c + (int64_t)i * cp.c_stride_bytes[2])[c16] = kv[u];
        reinterpret_cast<uint4*>(gh.v_c + (int64_t)i * cp.c_stride_bytes[2])[c16] = vv[u];
      }
    }
  }
}


// ---------------------------------------------------------------------------------------------------------
constexpr int SEL_CLUSTER = 8;

template <int SW, int KPT, int CS, bool RAW = false>
cudaError_t launch_select_topk_shape(const SelectParams& p, bool pdl, cudaStream_t st, const FoldOf<RAW>& fold = {}) {
  const size_t smem = RAW ? (size_t)((p.Lmax - p.b + CS - 1) / CS + p.window) * 4 : 0;
  if constexpr (RAW) {
    static SmemConfig configured;
    const cudaError_t e = configure_smem(reinterpret_cast<const void*>(select_topk_kernel<SW, KPT, CS, RAW>), smem, configured, false);
    if (e != cudaSuccess) return e;
  }
  int ctas = CS;
  if constexpr (RAW) ctas += fold.ctas;
  LaunchConfig lc(dim3(ctas, p.Hkv, p.B), 32 * SW, smem, st);
  if (CS > 1) lc.cluster(CS);
  if (pdl) lc.after_start_of_previous();
  return cudaLaunchKernelEx(&lc.cfg, select_topk_kernel<SW, KPT, CS, RAW>, p, fold);
}

// Candidates in the registers of one CTA up to 8192 per head; beyond that, for up to a quarter as many heads as SMs (two waves
// of clusters), in those of a cluster of eight CTAs (up to 65536), else again of one CTA, of 1024 threads (up to 32768); in
// global memory where neither fits. (30000 candidates: 32 heads 16.5 us with clusters, 39 without; 128 heads 61 and 39.) Tuning::select forces one CTA (1) or a cluster (2) per head.
cudaError_t launch_topk(const SelectParams& p, bool pdl, cudaStream_t st) {
  const int cand = p.Lmax - p.b, forced = tuning().select;
  const bool few = (long long)p.B * p.Hkv * 4 <= sm_count();
  if (forced != 2) {
    if (cand <= 512) return launch_select_topk_shape<8, 2, 1>(p, pdl, st);
    if (cand <= 1536) return launch_select_topk_shape<8, 6, 1>(p, pdl, st);
    if (cand <= 3072) return launch_select_topk_shape<16, 6, 1>(p, pdl, st);
    if (cand <= 5120) return launch_select_topk_shape<16, 10, 1>(p, pdl, st);
    if (cand <= 8192) return launch_select_topk_shape<16, 16, 1>(p, pdl, st);
    if (!few || forced == 1) {
      if (cand <= 16384) return launch_select_topk_shape<32, 16, 1>(p, pdl, st);
      if (cand <= 32768) return launch_select_topk_shape<32, 32, 1>(p, pdl, st);
    }
  }
  if (forced != 1) {
    if (cand <= SEL_CLUSTER * 4096) return launch_select_topk_shape<16, 8, SEL_CLUSTER>(p, pdl, st);
    if (cand <= SEL_CLUSTER * 8192) return launch_select_topk_shape<16, 16, SEL_CLUSTER>(p, pdl, st);
  }
  select_topk_global_kernel<<<dim3(p.Hkv, p.B), SELG_THREADS, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_gather(const CompactParams& p, bool pdl, cudaStream_t st) {
  if (p.n_keep_max <= 0) return cudaSuccess;
  const int rows_per_block = (256 / (p.row_bytes / 16)) * CP_ROWS_ALONE;
  LaunchConfig lc(dim3((p.n_keep_max + rows_per_block - 1) / rows_per_block, p.Hkv, p.B), 256, 0, st);
  if (pdl) lc.after_start_of_previous();
  return cudaLaunchKernelEx(&lc.cfg, compact_kv_kernel, p);
}

template <int SW, int KPT, bool RAW>
cudaError_t launch_select_gather(const cudaLaunchConfig_t& cfg, const SelectParams& p, const CompactParams& cp, const FoldOf<RAW>& fold) {
  static SmemConfig configured;
  auto kern = select_gather_kernel<SW, KPT, RAW>;
  const cudaError_t e = configure_smem(reinterpret_cast<const void*>(kern), cfg.dynamicSmemBytes, configured, false);
  return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, kern, p, cp, fold);
}

template <bool RAW>
cudaError_t launch_fused(const SelectParams& p, const CompactParams& cp, const FoldOf<RAW>& fold, cudaStream_t st) {
  int folds = 0;
  if constexpr (RAW) folds = fold.ctas;
  const int R = gather_ctas(p.B, p.Hkv, p.n_keep_max, folds);
  LaunchConfig lc(dim3((unsigned)R + folds, p.Hkv, p.B), 1024, (size_t)((p.n_keep_max + R - 1) / R + 1 + (RAW ? raw_axis_floats(p.Lmax, p.b, p.window) : 0)) * 4, st);
  if (tuning().pdl != 0) lc.after_start_of_previous();       // never releases its own dependents early
  const int cand = p.Lmax - p.b;
  if (cand <= 512) return launch_select_gather<8, 2, RAW>(lc.cfg, p, cp, fold);
  if (cand <= 1536) return launch_select_gather<8, 6, RAW>(lc.cfg, p, cp, fold);
  if (cand <= 3072) return launch_select_gather<16, 6, RAW>(lc.cfg, p, cp, fold);
  if (cand <= 5120) return launch_select_gather<16, 10, RAW>(lc.cfg, p, cp, fold);
  return launch_select_gather<16, 16, RAW>(lc.cfg, p, cp, fold);
}

}  // namespace

cudaError_t launch_select_topk(const SelectParams& p, cudaStream_t st) { return launch_topk(p, false, st); }

cudaError_t launch_compact(const CompactParams& p, cudaStream_t st) { return launch_gather(p, false, st); }

// Whether selection and gather run as one launch: a head's candidates must fit the registers of a CTA's selecting warps, and
// there are fewer heads than SMs (see select_gather_kernel). Otherwise the two kernels run one after the other.
bool select_compact_is_fused(int B, int Hkv, int Lmax, int b, int n_keep_max) {
  const int cand = Lmax - b;
  return cand >= 1 && cand <= 8192 && n_keep_max >= 1 && (long long)B * Hkv <= sm_count() && tuning().select == 0;
}

// CTAs per head: fill the SMs, but leave every CTA at least 64 rows to copy.
int gather_ctas(int B, int Hkv, int n_keep_max, int folds) {
  long long R = sm_count() / ((long long)B * Hkv) - folds;
  if (R > n_keep_max / 64) R = n_keep_max / 64;
  if (tuning().splits > 0) R = tuning().splits;
  return R > 16 ? 16 : (R < 1 ? 1 : (int)R);
}

cudaError_t launch_select_compact(const SelectParams& p, const CompactParams& cp, cudaStream_t st) {
  const bool pdl = tuning().pdl != 0;
  if (!select_compact_is_fused(p.B, p.Hkv, p.Lmax, p.b, p.n_keep_max)) {
    SelectParams alone = p;
    alone.gather_follows = p.n_keep_max > 0 ? 1 : 0;
    const cudaError_t e = launch_topk(alone, pdl, st);
    return e != cudaSuccess ? e : launch_gather(cp, pdl, st);
  }
  return launch_fused<false>(p, cp, NoFold{}, st);
}

cudaError_t launch_pool_select_compact(const SelectParams& p, const CompactParams& cp, const FoldParams& fold, cudaStream_t st) {
  if (select_compact_is_fused(p.B, p.Hkv, p.Lmax, p.b, p.n_keep_max)) return launch_fused<true>(p, cp, fold, st);
  const bool pdl = tuning().pdl != 0;
  SelectParams alone = p;
  alone.gather_follows = 1;
  FoldParams f = fold;
  if (f.ctas > 0) f.ctas = SEL_CLUSTER;
  const cudaError_t e = p.Lmax - p.b <= SEL_CLUSTER * 4096 ? launch_select_topk_shape<16, 8, SEL_CLUSTER, true>(alone, pdl, st, f)
                                                           : launch_select_topk_shape<16, 16, SEL_CLUSTER, true>(alone, pdl, st, f);
  return e != cudaSuccess ? e : launch_gather(cp, pdl, st);
}

// Selection by a cluster per head, which can pool and fold too: more candidates than a CTA holds, few heads (see launch_topk).
bool select_is_clustered(int B, int Hkv, int Lmax, int b, int n_keep_max) {
  const int cand = Lmax - b;
  return cand > 8192 && cand <= SEL_CLUSTER * 8192 && (long long)B * Hkv * 4 <= sm_count() && n_keep_max >= 1 && tuning().select == 0;
}

}  // namespace sdllm
