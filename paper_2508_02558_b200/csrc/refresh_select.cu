// Refresh step without its attention: mean-query saliency, pooling, top-k and gather of one (sequence, KV head) by one cluster of
// CTAs (Algorithm 1 from "qbar <- Mean(Q_b)" to the cache store), in one launch that runs BESIDE the attention kernel.
//
// The kept entries depend on the logits' means alone, not on the softmax, so nothing here has to wait for the attention; in a chain
// of the two a refresh of 32 heads x 1280 keys took 10 us of attention and 10 of selection and gather. For 10 MB of keys a second
// product K Q^T is cheap: K comes from L2 the second time. Whole refreshes, one after the other and beside: 32 heads x 300 / 1280 /
// 3100 keys 13.0 / 21.6 / 33.2 us and 11.0 / 17.6 / 30.0; 8 x 1280 15.0 and 12.0; 64 x 1280 28.6 and 21.9; 74 x 1280 31.1 and 23.6. What is
// left is a chain: 2 us to start behind the attention's first CTAs, 4 for the scores, 5 for the selection, 2.5 for the gather.
//   scores   the CTAs of the cluster share the head's tiles of 128 keys: TMA, S^T [128 keys x N queries] = K_tile Q^T (tcgen05), and
//            the thread that owns a key adds its logits up in the order of attn_kt.cu, so that the scores are that kernel's bit for
//            bit. They go into the shared memory of every CTA of the cluster, 4 bytes per key, counted by an mbarrier of the receiver.
//   the rest select_common.cuh: every CTA selects for itself, keeps its share of the list and copies its rows.
// The launch in front must let this one start only once it has seen everything before it complete, and writes nothing that is read
// here; this kernel ends only behind that one's end.
// Twelve warps of at most 56 registers and less than 120 KB leave room for a CTA of attn_kt.cu on the same SM (registers are
// allotted per SM quarter: its six warps take up to 10752 of 16384 there; with sixteen warps of 64 nothing ran beside anything).
// Every mbarrier wait is bounded; on expiry the CTA sets an abort flag, records a code in the status word, sends its peers the scores they
// count on all the same, waits at a second cluster barrier until theirs are on their way and for the bytes themselves (a CTA must not
// leave while a peer still writes to it), and runs to its end.
#include <cuda.h>
#include <string.h>

#include "fold.cuh"
#include "kt_params.cuh"
#include "tuning.cuh"
#include "umma_host.cuh"

namespace sdllm {
using namespace dev;
namespace {

#include "kt_common.cuh"
#include "select_common.cuh"

constexpr int RS_THREADS = 384, RS_SLOTS = 2, RS_SW = 8;
struct ScoreMaps {
  CUtensorMap q, k;
};

template <int D>
struct ScoreShape {
  static constexpr int H = D / 64, HALF = 128 * 128, TILE = H * HALF, QBYTES = H * 32 * 128;
  static constexpr int STAGES = gather_stages(RS_THREADS, RS_SLOTS * TILE);      // (the gather's stages lie over the ring)
  static constexpr size_t FIXED = 1024 /*alignment slack*/ + RS_SLOTS * TILE + QBYTES;
};

template <int D, int KPT>
__global__ void __launch_bounds__(RS_THREADS, 3) score_select_kernel(const __grid_constant__ ScoreMaps tm, const AttnParams p, const SelectParams sp,
                                                                     const CompactParams cp) {
  using Sh = ScoreShape<D>;
  constexpr int H = Sh::H, HALF = Sh::HALF, TILE = Sh::TILE, NS = RS_SLOTS, SW = RS_SW, NT = RS_THREADS;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(16) SelectShared<SW, 1> sh;
  __shared__ __align__(8) uint64_t bars_s[NS + 7];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x, R = gridDim.x, g = blockIdx.y, bi = blockIdx.z, N = p.M;
  volatile int* abort_flag = &abort_s;
  const uint32_t raw_addr = smem_u32(smem_raw);
  unsigned char* ring = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  unsigned char* q_s = ring + NS * TILE;
  int32_t* kept_s = reinterpret_cast<int32_t*>(q_s + Sh::QBYTES);
  float* raw_s = reinterpret_cast<float*>(kept_s + (sp.n_keep_max + R - 1) / R + 1);
  const uint32_t bars = smem_u32(bars_s);
  auto BAR = [&](int i) { return bars + 8u * (uint32_t)i; };
  constexpr int FULL = 0, S_FULL = NS, S_EMPTY = NS + 2, DRAIN = NS + 4, Q_FULL = NS + 5, SCORES = NS + 6;

  const int len = p.n1_per_seq ? __ldcg(p.n1_per_seq + bi) : p.n1_max, off = __ldcg(sp.block_off + bi);
  // The head's tiles, shared out evenly; with one sequence by the longest length, so that nothing waits for the length to load.
  const int tiles = (min(max(p.B == 1 ? p.n1_max : len, 0), p.n1_max) + 127) / 128, t0 = r * tiles / R, nt = (r + 1) * tiles / R - t0;
  int loads = 0;                                       // tiles whose load is under way (the lane that issues)
  auto load = [&](int t) {
    mbar_expect_tx(BAR(FULL + t % NS), (uint32_t)TILE);
    for (int hh = 0; hh < H; ++hh) tma_load_4d(smem_u32(ring + (t % NS) * TILE + hh * HALF), &tm.k, BAR(FULL + t % NS), hh * 64, (t0 + t) * 128, g, bi);
    loads = t + 1;
  };
  if (warp == 4) {
    if (elect_one()) {
      prefetch_tmap(&tm.k); prefetch_tmap(&tm.q);
      for (int i = 0; i < NS; ++i) mbar_init(BAR(FULL + i), 1);
      for (int i = 0; i < 2; ++i) { mbar_init(BAR(S_FULL + i), 1); mbar_init(BAR(S_EMPTY + i), 4); }
      mbar_init(BAR(DRAIN), 1);
      mbar_init(BAR(Q_FULL), 1);
      mbar_init(BAR(SCORES), 1);
      abort_s = 0;
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      if (nt > 0) {
        mbar_expect_tx(BAR(Q_FULL), (uint32_t)(H * N * 128));
        for (int hh = 0; hh < H; ++hh) tma_load_4d(smem_u32(q_s + hh * 32 * 128), &tm.q, BAR(Q_FULL), hh * 64, 0, g * p.G, bi);
      }
      for (int t = 0; t < nt && t < NS; ++t) load(t);
    }
    __syncwarp();
    tmem_alloc(smem_u32(&tmem_slot), 64);
    tmem_relinquish();
  }
  sh.clear(tid, NT);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive_relaxed();                            // "this CTA runs, its barriers are set up"; waited for before a peer is written to
  const uint32_t tmem_base = tmem_slot;
  const int L = min(max(len, 0), p.n1_max);
  const HeadPlace h = place_head(sp, L, off);
  const RawAxis axis(sp, h);
  if (tid == 0) mbar_expect_tx(BAR(SCORES), (uint32_t)h.C * 4u);      // the scores that come from all CTAs of the cluster, this one included
  axis.clear_ends(raw_s, h.C, tid, NT);

  // ======================================= scores =======================================
  if (warp == 4) {
    const bool leader = elect_one();
    bool ok = nt > 0 && wait_bar_warp(BAR(Q_FULL), 0, abort_flag, p.status, 16, p.wait_cycles);
    const uint64_t qd = smem_desc(smem_u32(q_s), 16u, 1024u);
    const uint32_t idesc = kt_idesc(32, false, false);
    for (int t = 0; t < nt && ok; ++t) {
      if (t >= 1 && t - 1 + NS < nt) {                 // the slot of tile t - 1 is free once its S^T is there
        if (!wait_bar_warp(BAR(S_FULL + ((t - 1) & 1)), ((t - 1) >> 1) & 1, abort_flag, p.status, 17, p.wait_cycles)) { ok = false; break; }
        if (leader) load(t - 1 + NS);
      }
      if (!wait_bar_warp(BAR(FULL + t % NS), (t / NS) & 1, abort_flag, p.status, 18, p.wait_cycles)) { ok = false; break; }
      if (t >= 2 && !wait_bar_warp(BAR(S_EMPTY + (t & 1)), ((t - 2) >> 1) & 1, abort_flag, p.status, 19, p.wait_cycles)) { ok = false; break; }
      tc_fence_after();
      const uint64_t kd = smem_desc(smem_u32(ring + (t % NS) * TILE), 16u, 1024u);
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          mma_ss(tmem_base + (t & 1) * 32, kd + (((ks >> 2) * HALF + (ks & 3) * 32) >> 4), qd + (((ks >> 2) * (32 * 128) + (ks & 3) * 32) >> 4), idesc, ks > 0 ? 1u : 0u);
        tc_commit(BAR(S_FULL + (t & 1)));
      }
      __syncwarp();
    }
  } else if (warp < 4) {
    const int row = warp * 32 + lane;
    bool ok = true;                                    // (a warp whose wait gave up still sends what its peers count on)
    for (int t = 0; t < nt; ++t) {
      ok = ok && wait_bar_warp(BAR(S_FULL + (t & 1)), (t >> 1) & 1, abort_flag, p.status, 20, p.wait_cycles);
      tc_fence_after();
      float a = 0.f;
      if (ok) {
        uint32_t sv[32];
        tmem_ld32(tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t & 1) * 32, sv);
        tc_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(S_EMPTY + (t & 1)));
        float a4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (c < N) a4[c & 3] += __uint_as_float(sv[c]);
        a = ((a4[0] + a4[1]) + (a4[2] + a4[3])) * (p.scale / (float)N);
      }
      if (t == 0) cluster_wait_acquire();
      const int pos = (t0 + t) * 128 + row, c = pos < h.o ? pos : pos - h.b;
      if (c < h.C && (pos < h.o || c >= h.o))
        for (int peer = 0; peer < R; ++peer)
          st_async_f1(map_to_cta(smem_u32(raw_s + axis.at(c)), (uint32_t)peer), map_to_cta(BAR(SCORES), (uint32_t)peer), a);
    }
  }
  if (warp >= 4 || nt == 0) cluster_wait_acquire();    // (every thread passes the barrier once)
  cluster_arrive_relaxed();                            // "this CTA's scores are on their way"
  tc_fence_before();
  wait_merge(BAR(SCORES), abort_flag, p.status, p.wait_cycles);      // the head's scores are here
  __syncthreads();
  if (*abort_flag) {                                   // a wait gave up, in whichever warp: what is under way lands first
    if (warp == 4 && nt > 0) {
      drain_mmas(BAR(DRAIN));
      drain_loads(BAR(FULL), loads, NS);               // (the lane that issued them knows their number)
      drain_bar(BAR(Q_FULL), 0);
      __syncwarp();
    }
    cluster_wait_acquire();                            // a slower peer may still be sending: this CTA goes on, and leaves, when all is here
    drain_bar(BAR(SCORES), 0);
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 4) tmem_dealloc(tmem_base, 64);

  // ======================================= pooling, selection, gather =======================================
  const int kpt = min((h.C + 32 * SW - 1) / (32 * SW), KPT);
  const int c0 = warp * 32 * kpt + lane;
  const int64_t head = bi * p.Hkv + g;
  int32_t* out = sp.kept_idx + head * sp.n_keep_max;
  // this CTA's share: the kept entries [i_lo, i_hi) and the empty ones [z_lo, z_hi) of the head's list (R <= 8)
  const int pad = sp.n_keep_max - h.kept;
  const int i_lo = r * h.kept / R, i_hi = (r + 1) * h.kept / R;
  const int z_lo = h.kept + r * pad / R, z_hi = h.kept + (r + 1) * pad / R;
  const GatherHead gh = gather_head(cp, bi, g);
  if (warp < SW) {
    uint32_t key[KPT];
    pool_keys(key, axis, raw_s, h.C, kpt, c0);
    select_head<SW, KPT, 1>(h, key, c0, sh, 0, [&](int w, int c) {
      if (w >= i_lo && w < i_hi) kept_s[w - i_lo] = c < h.o ? c : c + h.b;
    });
  } else {
    const int t = tid - 32 * SW, nt = NT - 32 * SW;    // what does not wait for the selection
    if (g == 0 && r == 0 && t == 0) sp.kept_cnt[bi] = h.kept;
    write_pooled(sp, raw_s, h, head, r, R, t, nt);
    write_empty_entries(cp, gh, out, z_lo, z_hi, t, nt);
  }
  __syncthreads();
  for (int i = i_lo + tid; i < i_hi; i += NT) out[i] = kept_s[i - i_lo];
  gather_rows<NT, Sh::STAGES>(cp, gh, ring, kept_s, i_lo, i_hi);
  if (!*abort_flag) cluster_wait_acquire();            // (every thread passes the second barrier once)
  grid_dependency_wait();                              // this launch must not be over before the one in front of it is
}

template <int D, int KPT>
cudaError_t launch_shape(const ScoreMaps& tm, const AttnParams& p, const SelectParams& sp, const CompactParams& cp, int R, cudaStream_t st) {
  auto kern = score_select_kernel<D, KPT>;
  static SmemConfig configured;
  // (more than half of what a CTA of attn_kt.cu leaves over: two of these on one SM would only stand in each other's way)
  size_t smem = ScoreShape<D>::FIXED + (size_t)((sp.n_keep_max + R - 1) / R + 1 + raw_axis_floats(sp.Lmax, sp.b, sp.window)) * 4;
  if (smem < 97 * 1024) smem = 97 * 1024;
  LaunchConfig lc(dim3(R, p.Hkv, p.B), RS_THREADS, smem, st);
  const cudaError_t e = configure_smem(reinterpret_cast<const void*>(kern), lc.cfg.dynamicSmemBytes, configured, true);
  if (e != cudaSuccess) return e;
  lc.cluster(R);
  if (tuning().pdl != 0) lc.after_start_of_previous();
  return cudaLaunchKernelEx(&lc.cfg, kern, tm, p, sp, cp);
}

template <int D>
cudaError_t launch_d(const ScoreMaps& tm, const AttnParams& p, const SelectParams& sp, const CompactParams& cp, int R, cudaStream_t st) {
  // (1537 to 2304 candidates with twelve per thread instead of nine lost 2 to 6 % to the two parts of the refresh with 16 to 32 heads)
  const int cand = sp.Lmax - sp.b;
  if (cand <= 512) return launch_shape<D, 2>(tm, p, sp, cp, R, st);
  if (cand <= 1536) return launch_shape<D, 6>(tm, p, sp, cp, R, st);
  if (cand <= 2304) return launch_shape<D, 9>(tm, p, sp, cp, R, st);
  return launch_shape<D, 12>(tm, p, sp, cp, R, st);
}

}  // namespace

// At least two CTAs per head, launched as a cluster. (A form of one CTA per head without a cluster launch raised "an illegal instruction"
// once, at 128 units; its cause is not known. Only there did barrier.cluster, mapa and st.async run outside a cluster launch.)
bool score_select_supported(int D, int M, int units, int cand) {
  return (D == 64 || D == 128) && M <= 32 && cand >= 1 && cand <= 3072 && 2 * units <= sm_count();
}

cudaError_t launch_score_select(const AttnParams& p, const SelectParams& sp, const CompactParams& cp, int D, cudaStream_t st) {
  ScoreMaps tm;
  memset(&tm, 0, sizeof(tm));
  if (!umma_make_map(&tm.q, p.q, D, p.b, p.Hq, p.B, p.q_stride, p.b, p.G) || !umma_make_map(&tm.k, p.k1, D, p.n1_max, p.Hkv, p.B, p.k1_stride, 128, 1))
    return cudaErrorInvalidValue;
  long long R = sm_count() / ((long long)p.B * p.Hkv);
  if (R > 8) R = 8;
  if (R < 2) return cudaErrorInvalidValue;
  return D == 128 ? launch_d<128>(tm, p, sp, cp, (int)R, st) : launch_d<64>(tm, p, sp, cp, (int)R, st);
}

}  // namespace sdllm
