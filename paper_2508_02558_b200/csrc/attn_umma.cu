// bf16 block-query attention on the tensor cores (tcgen05), queries on the accumulator rows, one softmax warpgroup: the attention
// pass in front of the probability saliency (attn_prob.cu), which needs the rows' log-sum-exp. Every other call goes to attn_kt.cu and
// attn_pair.cu; this kernel stays because that saliency ranks keys by differences as small as the rounding of exp2(S - log-sum-exp),
// and the order of the sums behind the log-sum-exp is this kernel's.
//
// One CTA owns (sequence, KV head, 128-row tile of the head's b*G query rows, key split) and streams its share of the sequence's
// K/V once. Warp roles (256 threads):
//   warp 0      TMA producer: K and V tiles (128-byte swizzle) into a shared-memory ring, one mbarrier pair per slot
//   warp 1      tcgen05.mma issuer: S = Q K^T (A, B from shared memory) into TMEM, then
//               O_tile = P V with P read from TMEM (A) and V from shared memory (B, MN-major)
//   warps 2-5   softmax: each thread owns one of the 128 accumulator rows (TMEM lane), reads its S row with
//               tcgen05.ld, keeps the running max / sum and writes P (bf16) over S in TMEM; O accumulates in TMEM
//               across the tiles and is rescaled in place only when a row's maximum grows by more than 2^8
//   warps 6-7   help on the way out only
// When b*G <= 64 the query rows are replicated R = 2 or 4 times along the 128 accumulator rows and every replica
// takes its own slice of each key tile, so all four softmax warps work; the replicas are merged like key splits, inside the CTA
// through shared memory. Key splits leave (max, sum, O) partials in the workspace. While that is little, the last CTA of a
// (sequence, KV head, row tile) to finish - found with one atomic counter, nobody waits - merges them and writes the output;
// larger volumes are merged by a second small launch spread over the whole GPU.
//
// Every wait on an mbarrier is bounded. On expiry the thread sets an abort flag that all other waits poll, records a
// code in the status word and the CTA runs to its end (freeing its TMEM); the outputs of that call are then invalid.
#include <cuda.h>
#include <string.h>

#include "attn_device.cuh"
#include "tuning.cuh"
#include "umma_host.cuh"

namespace sdllm {
using namespace dev;
namespace {

constexpr int UM_THREADS = 256;
constexpr int UM_STAGES = 3;

struct UmmaMaps {
  CUtensorMap q, k, v;
};

struct UmmaParams {
  AttnParams a;
  int KT;            // keys of a tile (64 or 128)
  int R;             // replicas of the query rows along the 128 accumulator rows (1, 2, 4)
  int row_tiles;     // 128-row tiles of the b*G rows
  int heads_rt;      // query heads per row tile
  int fused_tail;    // 1: the last CTA of a unit merges the key splits; 0: umma_tail_kernel does
  int lpt;           // 1: grid z counts the sequences from the longest to the shortest (several waves of ragged work)
};

#include "umma_ptx.cuh"

// Merge of the key-split partials of S (row, float4 column) slots of a unit and the final stores. slot[s] < 0 marks
// an unused entry. The partials are read in batches of MB per slot with the loads of all slots and of the whole batch
// in flight together (one L2 latency per batch) and folded with a running maximum, so that four splits cost a single
// round trip for everything a thread merges.
template <int D, int MB, int S>
__device__ __forceinline__ void merge_slots(const AttnParams& p, int64_t unit, int bi, int g, int rt, const int (&slot)[S]) {
  constexpr int D4 = D / 4;
  const int P = p.splits;
  const int prt = min(p.M, 128);                      // rows of one partial
  const float2* ml_base = reinterpret_cast<const float2*>(p.part_ml) + unit * P * prt;
  const float4* po_base = reinterpret_cast<const float4*>(p.part_o + unit * P * prt * D);
  float4 acc[S];
  float l[S], m_run[S];
  int m_local[S], d4[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    acc[s] = make_float4(0.f, 0.f, 0.f, 0.f); l[s] = 0.f; m_run[s] = -INFINITY;
    const int sl = max(slot[s], 0);
    m_local[s] = sl / D4; d4[s] = sl - m_local[s] * D4;
  }
  for (int p0 = 0; p0 < P; p0 += MB) {
    float2 x[S][MB];
    float4 o[S][MB];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int u = 0; u < MB; ++u) {
        const int pi = min(p0 + u, P - 1);
        x[s][u] = __ldcg(ml_base + (int64_t)pi * prt + m_local[s]);
        o[s][u] = __ldcg(po_base + ((int64_t)pi * prt + m_local[s]) * D4 + d4[s]);
      }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      float bm = m_run[s];
#pragma unroll
      for (int u = 0; u < MB; ++u)
        if (p0 + u < P && x[s][u].y != 0.f) bm = fmaxf(bm, x[s][u].x);
      const float a = (bm == -INFINITY) ? 1.f : fast_exp2(m_run[s] - bm);    // 0 on the first batch with data
      acc[s].x *= a; acc[s].y *= a; acc[s].z *= a; acc[s].w *= a; l[s] *= a;
      m_run[s] = bm;
#pragma unroll
      for (int u = 0; u < MB; ++u) {
        if (p0 + u >= P || x[s][u].y == 0.f) continue;
        const float w = fast_exp2(x[s][u].x - bm);
        l[s] = fmaf(x[s][u].y, w, l[s]);
        acc[s].x = fmaf(o[s][u].x, w, acc[s].x); acc[s].y = fmaf(o[s][u].y, w, acc[s].y);
        acc[s].z = fmaf(o[s][u].z, w, acc[s].z); acc[s].w = fmaf(o[s][u].w, w, acc[s].w);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    if (slot[s] < 0) continue;
    const float inv = l[s] > 0.f ? 1.f / l[s] : 0.f;
    const int m = rt * 128 + m_local[s];
    const int hg = m / p.b, i = m - hg * p.b;
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (int64_t)bi * p.o_stride[0] +
                         (int64_t)(g * p.G + hg) * p.o_stride[1] + (int64_t)i * p.o_stride[2] + d4[s] * 4;
    uint2 w2;
    w2.x = pack_bf16(acc[s].x * inv, acc[s].y * inv);
    w2.y = pack_bf16(acc[s].z * inv, acc[s].w * inv);
    *reinterpret_cast<uint2*>(out) = w2;
    if (d4[s] == 0 && p.lse) p.lse[((int64_t)bi * p.Hq + g * p.G + hg) * p.b + i] = (m_run[s] + log2f(l[s])) * kLn2;
  }
}

// Deferred tail (large partial volumes): one launch that merges the key splits, one thread per (row, float4 column).
template <int D>
__global__ void __launch_bounds__(256) umma_tail_kernel(const UmmaParams up) {
  const AttnParams& p = up.a;
  grid_dependency_wait();
  grid_launch_dependents();
  constexpr int D4 = D / 4;
  const int64_t slot = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int d4 = (int)(slot % D4);
  const int64_t r = slot / D4;
  const int m_local = (int)(r % 128);
  const int64_t unit = r / 128;
  if (unit >= (int64_t)p.B * p.Hkv * up.row_tiles) return;
  const int rt = (int)(unit % up.row_tiles);
  const int64_t bg = unit / up.row_tiles;
  const int g = (int)(bg % p.Hkv), bi = (int)(bg / p.Hkv);
  if (m_local >= min(p.M - rt * 128, 128)) return;
  const int one[1] = {m_local * D4 + d4};
  merge_slots<D, 8, 1>(p, unit, bi, g, rt, one);
}

template <int D>
__global__ void __launch_bounds__(UM_THREADS, 1) attn_umma_bf16_kernel(const __grid_constant__ UmmaMaps tm, const UmmaParams up) {
  constexpr int H = D / 64;            // 128-byte column halves of a row
  constexpr int NS = UM_STAGES;
  constexpr int NCH = 4;               // 32-column chunks of a key tile
  constexpr uint32_t S_STRIDE = 128;   // TMEM columns: the two S/P buffers, then the O accumulator
  constexpr uint32_t O_COL = 2 * S_STRIDE;
  constexpr uint32_t TMEM_COLS = 512;
  constexpr int CTRL = 1024;           // control block: barriers, flags
  const AttnParams& p = up.a;
  extern __shared__ unsigned char smem_raw[];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int KT = up.KT, R = up.R;
  const int rows_rep = 128 / R;
  int bi = blockIdx.z;
  if (up.lpt) {
    grid_dependency_wait();                            // the lengths may come from the kernel in front
    bi = sequence_of_rank(p.n1_per_seq, p.B, blockIdx.z);
  }
  const int g = blockIdx.y / up.row_tiles, rt = blockIdx.y - g * up.row_tiles;
  const int split = blockIdx.x;
  const int tiles = (p.n1_max + KT - 1) / KT;
  const int t_begin = (int)(((long long)split * tiles) / p.splits);
  const int t_end = (int)(((long long)(split + 1) * tiles) / p.splits);
  const int M_rt = min(p.M - rt * 128, 128);          // valid query rows of this row tile (<= rows_rep when R > 1)

  // ---- shared memory carve-up (1024-byte aligned for the 128-byte swizzle) ----
  const uint32_t raw_addr = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t bars = smem_u32(smem);
  auto BAR = [&](int i) { return bars + 8u * (uint32_t)i; };
  const int Q_FULL = 0, FULL_K = 1, FULL_V = 1 + NS, EMPTY_K = 1 + 2 * NS, EMPTY_V = 1 + 3 * NS;
  const int S_FULL = 1 + 4 * NS, P_FULL = S_FULL + 2, PV_DONE = S_FULL + 4, DRAIN = S_FULL + 6;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 260);
  int* last_flag = reinterpret_cast<int*>(smem + 264);
  int* issued_s = reinterpret_cast<int*>(smem + 268);  // [2] tiles whose K / V loads are on their way (for an aborted CTA's way out)
  unsigned char* q_s = smem + CTRL;
  unsigned char* stage0 = q_s + H * 128 * 128;
  const int half_bytes = KT * 128;                     // one 64-column half of a K or V tile
  const int kv_bytes = H * half_bytes;                 // a whole K (or V) tile
  const int stage_bytes = 2 * kv_bytes;
  // The Q box (b rows x the row tile's heads) is loaded as many times as it fits into the 128 accumulator rows: every
  // replica starts on a copy, and rows past the valid ones hold real data whose results are simply not used. Only a box
  // that does not divide 128 leaves rows uncovered; those must not hold non-finite garbage and are cleared first.
  const int q_rows = p.b * up.heads_rt;
  const int q_copies = (128 % q_rows == 0) ? 128 / q_rows : R;
  const int q_step = (128 % q_rows == 0) ? q_rows : rows_rep;
  const bool zero_q = 128 % q_rows != 0 && q_rows < rows_rep;
  if (tid == 0) {                        // the descriptors live in the kernel parameters: fetch them while the CTA sets up
    prefetch_tmap(&tm.k); prefetch_tmap(&tm.v); prefetch_tmap(&tm.q);
  }

  // The producer lane sets the barriers up and, unless the Q tile has to be cleared first, starts the first loads
  // before the rest of the CTA is ready: the loads need nothing but the barriers.
  int n1 = 0;
  auto read_count = [&]() { n1 = min(max(p.n1_per_seq ? p.n1_per_seq[bi] : p.n1_max, 0), p.n1_max); };
  auto valid_keys = [&](int t) { return min(max(n1 - t * KT, 0), KT); };               // of tile t; 0: the tile is skipped
  int prod_it = 0, prod_t = t_begin;
  bool prod_ok = true, v_missing = false, q_issued = false;
  auto issue_q = [&]() {              // the Q tile (replicated R times along the accumulator rows)
    q_issued = true;
    mbar_expect_tx(BAR(Q_FULL), (uint32_t)(q_copies * H * q_rows * 128));
    for (int c = 0; c < q_copies; ++c)
      for (int h = 0; h < H; ++h)
        tma_load_4d(smem_u32(q_s + h * 128 * 128 + c * q_step * 128), &tm.q, BAR(Q_FULL), h * 64, 0,
                    g * p.G + rt * up.heads_rt, bi);
  };
  // issue loads for up to `limit` further tiles (producer lane only)
  auto produce = [&](int limit) {
    for (; prod_t < t_end && limit > 0 && prod_ok; ++prod_t) {
      if (valid_keys(prod_t) == 0) continue;
      const int it = prod_it, s = it % NS;
      const uint32_t ph = ((it / NS) - 1) & 1;
      const uint32_t kdst = smem_u32(stage0 + (size_t)s * stage_bytes), vdst = kdst + kv_bytes;
      if (it >= NS && !wait_bar(BAR(EMPTY_K + s), ph, abort_flag, p.status, 1, p.wait_cycles)) { prod_ok = false; break; }
      ++prod_it;
      mbar_expect_tx(BAR(FULL_K + s), (uint32_t)kv_bytes);
      for (int h = 0; h < H; ++h) tma_load_4d(kdst + h * half_bytes, &tm.k, BAR(FULL_K + s), h * 64, prod_t * KT, g, bi);
      if (it >= NS && !wait_bar(BAR(EMPTY_V + s), ph, abort_flag, p.status, 2, p.wait_cycles)) { prod_ok = false; v_missing = true; break; }
      mbar_expect_tx(BAR(FULL_V + s), (uint32_t)kv_bytes);
      for (int h = 0; h < H; ++h) tma_load_4d(vdst + h * half_bytes, &tm.v, BAR(FULL_V + s), h * 64, prod_t * KT, g, bi);
      --limit;
    }
  };

  if (tid == 0) {
    mbar_init(BAR(Q_FULL), 1);
    for (int s = 0; s < NS; ++s) {
      mbar_init(BAR(FULL_K + s), 1);
      mbar_init(BAR(FULL_V + s), 1);
      mbar_init(BAR(EMPTY_K + s), 1);
      mbar_init(BAR(EMPTY_V + s), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(S_FULL + i), 1);
      mbar_init(BAR(P_FULL + i), 4);
      mbar_init(BAR(PV_DONE + i), 1);
    }
    mbar_init(BAR(DRAIN), 1);
    *abort_flag = 0;
    *last_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    if (!zero_q) {
      grid_dependency_wait();          // the loads read what earlier kernels in the stream wrote
      read_count();
      issue_q();
      produce(NS);                     // the first NS slots are free: no waiting here
    }
  }
  if (zero_q)
    for (int i = tid; i < H * 128 * 128 / 16; i += UM_THREADS) reinterpret_cast<uint4*>(q_s)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (warp == 1) {                     // the MMA warp owns the tensor memory
    tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();              // everything below may read what earlier kernels in the stream wrote
  grid_launch_dependents();
  read_count();

  // softmax state of this thread's accumulator row (softmax warps only)
  float m_run = -INFINITY, l_run = 0.f;
  bool sm_ok = true;
  int sm_tiles = 0;

  if (warp == 0) {
    // ======================================= TMA producer =======================================
    if (lane == 0) {
      if (!q_issued) issue_q();
      produce(1 << 30);
      issued_s[0] = prod_it; issued_s[1] = prod_it - (v_missing ? 1 : 0);
    }
  } else if (warp == 1) {
    // ======================================= MMA issuer =======================================
    // warp-uniform, one elected lane issues (see attn_kt.cu)
    const bool leader = elect_one();
    const uint32_t idesc_pv = instr_desc(D, true);
    bool ok = true, have_q = false;
    int it = 0;
    int prev_mma = 0;                                // MMA width of the tile whose P V comes next: its keys rounded up to 16
    auto issue_pv = [&](int n_mma, int j) -> bool {
      const int s = j % NS, pb = j & 1;
      if (!wait_bar_warp(BAR(P_FULL + pb), (j >> 1) & 1, abort_flag, p.status, 4, p.wait_cycles)) return false;
      if (!wait_bar_warp(BAR(FULL_V + s), (j / NS) & 1, abort_flag, p.status, 5, p.wait_cycles)) return false;
      tc_fence_after();
      const uint32_t vsm = smem_u32(stage0 + (size_t)s * stage_bytes) + kv_bytes;
      const uint32_t a_t = tmem_base + (uint32_t)pb * S_STRIDE;
      const uint64_t vd = smem_desc(vsm, (uint32_t)half_bytes, 1024u);
      if (leader) {
        for (int ks = 0; ks < n_mma / 16; ++ks) mma_ts(tmem_base + O_COL, a_t + ks * 8, vd + ks * (2048 >> 4), idesc_pv, (j > 0 || ks > 0) ? 1u : 0u);
        tc_commit(BAR(PV_DONE + pb));  // two alternating barriers: a waiter is never a whole phase ahead of either
        tc_commit(BAR(EMPTY_V + s));
      }
      __syncwarp();
      return true;
    };
    for (int t = t_begin; t < t_end && ok; ++t) {
      const int n_mma = (valid_keys(t) + 15) & ~15;
      if (n_mma == 0) continue;
      const int s = it % NS, sb = it & 1;
      if (!wait_bar_warp(BAR(FULL_K + s), (it / NS) & 1, abort_flag, p.status, 7, p.wait_cycles)) { ok = false; break; }
      if (!have_q) {
        if (!wait_bar_warp(BAR(Q_FULL), 0, abort_flag, p.status, 3, p.wait_cycles)) { ok = false; break; }
        have_q = true;
      }
      tc_fence_after();
      const uint32_t ksm = smem_u32(stage0 + (size_t)s * stage_bytes);
      const uint32_t qsm = smem_u32(q_s);
      const uint32_t idesc_s = instr_desc(n_mma, false);
      const uint32_t d_t = tmem_base + (uint32_t)sb * S_STRIDE;
      const uint64_t qd = smem_desc(qsm, 16u, 1024u), kd = smem_desc(ksm, 16u, 1024u);
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          mma_ss(d_t, qd + (((ks >> 2) * (128 * 128) + (ks & 3) * 32) >> 4), kd + (((ks >> 2) * half_bytes + (ks & 3) * 32) >> 4), idesc_s, ks > 0 ? 1u : 0u);
        tc_commit(BAR(S_FULL + sb));
        tc_commit(BAR(EMPTY_K + s));
      }
      __syncwarp();
      if (it > 0 && !issue_pv(prev_mma, it - 1)) { ok = false; break; }
      prev_mma = n_mma;
      ++it;
    }
    if (ok && it > 0) ok = issue_pv(prev_mma, it - 1);
    // a CTA whose slice holds no valid key never used Q: its load must still have landed before the CTA retires
    if (ok && !have_q) ok = wait_bar_warp(BAR(Q_FULL), 0, abort_flag, p.status, 3, p.wait_cycles);
  } else if (warp < 6) {
    // ======================================= softmax warps =======================================
    const int q4 = warp & 3;                         // TMEM lane quadrant this warp may access
    const int row = q4 * 32 + lane;
    const int rep = row / rows_rep;                  // warp-uniform
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
    const int chunk_keys = KT / R;                   // key slice of a tile owned by this replica
    int it = 0;
    bool ok = true;
    for (int t = t_begin; t < t_end && ok; ++t) {
      const int nv = valid_keys(t), n_mma = (nv + 15) & ~15;
      if (nv == 0) continue;
      const int s = it % NS, sb = it & 1;
      // columns of this tile owned by this replica; a warp whose 32 accumulator rows all lie beyond the valid rows of
      // its replica owns nothing
      const bool idle = q4 * 32 - rep * rows_rep >= M_rt;
      const int c_lo = idle ? nv : min(rep * chunk_keys, nv), c_hi = min((rep + 1) * chunk_keys, nv);
      if (!wait_bar_warp(BAR(S_FULL + sb), (it >> 1) & 1, abort_flag, p.status, 9, p.wait_cycles)) { ok = false; break; }
      tc_fence_after();
      const uint32_t s_addr = lane_addr + (uint32_t)sb * S_STRIDE;
      // ---- the owned part of the S row. Chunks of 32 columns that are owned and valid as a whole go through the
      //      unrolled register path, all their loads in flight together; the one chunk the end of the slice may cut
      //      (cp) takes a small predicated path of its own, so the common code stays short ----
      const int cf_lo = c_lo >> 5, cf_hi = c_hi >> 5;          // full chunks [cf_lo, cf_hi); c_lo is a multiple of 32
      const int cp = (c_hi & 31) && c_lo < c_hi ? cf_hi : -1;  // partial chunk, if any
      uint32_t sv[NCH][32];
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if (c >= cf_lo && c < cf_hi) tmem_ld32(s_addr + c * 32, sv[c]);
      uint32_t tv[32];
      if (cp >= 0) tmem_ld32(s_addr + cp * 32, tv);
      tc_wait_ld();
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if (c >= cf_lo && c < cf_hi) {
          float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int i = 0; i < 32; ++i) m4[i & 3] = fmaxf(m4[i & 3], __uint_as_float(sv[c][i]));
          mx = fmaxf(mx, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
        }
      if (cp >= 0) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (cp * 32 + i >= c_lo && cp * 32 + i < c_hi) mx = fmaxf(mx, __uint_as_float(tv[i]));
      }
      // ---- running maximum: O (in TMEM) and l are rescaled only when the maximum grows by more than 2^8, so P stays
      //      below 2^8 and the accumulator is touched on very few tiles ----
      const float m_new = fmaxf(m_run, mx * p.scale_log2);
      const bool grow = m_new > m_run + 8.f;          // also true on the first finite maximum
      float alpha = 1.f;
      if (grow) {
        alpha = fast_exp2(m_run - m_new);             // 0 when m_run is -inf
        m_run = m_new;
        l_run *= alpha;
      }
      if (it > 0 && __any_sync(0xffffffffu, grow)) {
        // every PV issued so far must have landed before the rows are rewritten; PV of this tile waits for our arrive
        if (!wait_bar_warp(BAR(PV_DONE + ((it - 1) & 1)), ((it - 1) >> 1) & 1, abort_flag, p.status, 8, p.wait_cycles)) { ok = false; break; }
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < D / 16; ++c) {
          uint32_t ov[16];
          tmem_ld16(lane_addr + O_COL + c * 16, ov);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
          tmem_st16(lane_addr + O_COL + c * 16, ov);
        }
      }
      const float mu = (m_run == -INFINITY) ? 0.f : m_run;
      // ---- P = exp2(S * scale_log2 - mu) as bf16 over the S columns; zero outside the owned slice ----
      float psum = 0.f;
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if (c >= cf_lo && c < cf_hi) {
          uint32_t pk[16];
          float ps4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float e0 = fast_exp2(fmaf(__uint_as_float(sv[c][2 * i]), p.scale_log2, -mu));
            const float e1 = fast_exp2(fmaf(__uint_as_float(sv[c][2 * i + 1]), p.scale_log2, -mu));
            ps4[i & 3] += e0 + e1;
            pk[i] = pack_bf16(e0, e1);
          }
          psum += (ps4[0] + ps4[1]) + (ps4[2] + ps4[3]);
          tmem_st16(s_addr + c * 16, pk);
        }
      if (cp >= 0) {
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int j0 = cp * 32 + 2 * i;
          const float e0 = (j0 >= c_lo && j0 < c_hi) ? fast_exp2(fmaf(__uint_as_float(tv[2 * i]), p.scale_log2, -mu)) : 0.f;
          const float e1 = (j0 + 1 >= c_lo && j0 + 1 < c_hi) ? fast_exp2(fmaf(__uint_as_float(tv[2 * i + 1]), p.scale_log2, -mu)) : 0.f;
          psum += e0 + e1;
          pk[i] = pack_bf16(e0, e1);
        }
        tmem_st16(s_addr + cp * 16, pk);
      }
      if (R > 1) {                                    // the other replicas' slices of this tile read as zero
        uint32_t zz[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) zz[i] = 0u;
#pragma unroll 1
        for (int c = 0; c * 32 < n_mma; ++c)
          if (!(c >= cf_lo && c < cf_hi) && c != cp) tmem_st16(s_addr + c * 16, zz);
      }
      l_run += psum;
      // ---- V rows past the source's count may hold anything: zero them so that 0 * V stays 0 ----
      if (nv < n_mma) {
        if (!wait_bar_warp(BAR(FULL_V + s), (it / NS) & 1, abort_flag, p.status, 10, p.wait_cycles)) { tc_wait_st(); ok = false; break; }   // (stores to tensor memory may be under way)
        unsigned char* vs = stage0 + (size_t)s * stage_bytes + kv_bytes;
        const int nz = (n_mma - nv) * H * 8;     // 16-byte chunks to clear
        for (int i = (warp - 2) * 32 + lane; i < nz; i += 128) {
          const int rr = nv + i / (H * 8), c = i % (H * 8);
          *reinterpret_cast<uint4*>(vs + (c >> 3) * half_bytes + rr * 128 + (((c & 7) ^ (rr & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
      }
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(P_FULL + sb));
      ++it;
    }
    sm_ok = ok; sm_tiles = it;
  }

  // ======================================= epilogue =======================================
  // The ring is idle now (every load was consumed), so it serves as scratch for the way out of TMEM:
  //   o_s [128][D] fp32, the float4 index XOR-swizzled by the row; ml_s [128]; lm_s [rows_rep].
  // Each accumulator row is weighted for the merge of the R replicas while it moves from TMEM to shared memory;
  // then consecutive threads store consecutive float4 of a row, so every global store is coalesced.
  const int64_t unit = (int64_t)(bi * p.Hkv + g) * up.row_tiles + rt;      // (sequence, KV head, row tile)
  if (warp >= 2 && warp < 6) {
    constexpr int D4 = D / 4;
    const int q4 = warp & 3;
    const int row = q4 * 32 + lane;
    const int rep = row / rows_rep, m_local = row - rep * rows_rep;
    float* o_s = reinterpret_cast<float*>(stage0);
    float2* ml_s = reinterpret_cast<float2*>(stage0 + 128 * D * 4);
    float2* lm_s = ml_s + 128;
    ml_s[row] = make_float2(m_run, l_run);
    asm volatile("bar.sync 2, 128;\n" ::: "memory");
    float mstar = -INFINITY;
    for (int r2 = 0; r2 < R; ++r2) {
      const float2 x = ml_s[r2 * rows_rep + m_local];
      if (x.y != 0.f) mstar = fmaxf(mstar, x.x);
    }
    float lsum = 0.f;
    for (int r2 = 0; r2 < R; ++r2) {
      const float2 x = ml_s[r2 * rows_rep + m_local];
      if (x.y != 0.f) lsum = fmaf(x.y, fast_exp2(x.x - mstar), lsum);
    }
    const float w = l_run != 0.f ? fast_exp2(m_run - mstar) : 0.f;       // this replica's weight in the merged row
    if (rep == 0) lm_s[m_local] = make_float2(mstar, lsum);
    // the finished accumulator row: TMEM -> weight -> shared memory, 32 columns at a time
    const bool have_o = sm_ok && sm_tiles > 0 &&
                        wait_bar_warp(BAR(PV_DONE + ((sm_tiles - 1) & 1)), ((sm_tiles - 1) >> 1) & 1, abort_flag, p.status, 6, p.wait_cycles);
    tc_fence_after();
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      uint32_t ov[32];
      if (have_o) {
        tmem_ld32(tmem_base + ((uint32_t)(q4 * 32) << 16) + O_COL + c * 32, ov);
        tc_wait_ld();
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) ov[i] = 0u;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *reinterpret_cast<float4*>(o_s + row * D + (((c * 8 + j) ^ (row & (D4 - 1))) << 2)) =
            make_float4(__uint_as_float(ov[4 * j]) * w, __uint_as_float(ov[4 * j + 1]) * w, __uint_as_float(ov[4 * j + 2]) * w,
                        __uint_as_float(ov[4 * j + 3]) * w);
    }
  }
  // all eight warps share the stores: consecutive threads take consecutive float4 of a row; a thread keeps its column
  // and walks down the rows, four rows per step with all their shared-memory reads in flight together
  constexpr int D4 = D / 4;
  const float* o_s = reinterpret_cast<const float*>(stage0);
  const float2* lm_s = reinterpret_cast<const float2*>(stage0 + 128 * D * 4) + 128;
  __syncthreads();
  const int st = tid;
  if (!*abort_flag) {
    const int d4 = st % D4, r_first = st / D4, r_step = UM_THREADS / D4;
    const int m_first = rt * 128;
    for (int mb = r_first; mb < M_rt; mb += 4 * r_step) {
      float4 acc[4];
      float2 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ml = min(mb + u * r_step, M_rt - 1);
        acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        x[u] = lm_s[ml];
        for (int r2 = 0; r2 < R; ++r2) {
          const int rr = r2 * rows_rep + ml;
          const float4 o = *reinterpret_cast<const float4*>(o_s + rr * D + ((d4 ^ (rr & (D4 - 1))) << 2));
          acc[u].x += o.x; acc[u].y += o.y; acc[u].z += o.z; acc[u].w += o.w;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ml = mb + u * r_step;
        if (ml >= M_rt) break;
        const int m = m_first + ml;                  // row within the KV head: m = head_in_group * b + i
        const int hg = m / p.b, i = m - hg * p.b;
        if (p.splits == 1) {
          const float inv = x[u].y > 0.f ? 1.f / x[u].y : 0.f;
          __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(p.out) + (int64_t)bi * p.o_stride[0] +
                             (int64_t)(g * p.G + hg) * p.o_stride[1] + (int64_t)i * p.o_stride[2] + d4 * 4;
          uint2 w2;
          w2.x = pack_bf16(acc[u].x * inv, acc[u].y * inv);
          w2.y = pack_bf16(acc[u].z * inv, acc[u].w * inv);
          *reinterpret_cast<uint2*>(o) = w2;
          if (d4 == 0 && p.lse) p.lse[((int64_t)bi * p.Hq + g * p.G + hg) * p.b + i] = (x[u].x + log2f(x[u].y)) * kLn2;
        } else {
          const int64_t prow = (unit * p.splits + split) * min(p.M, 128) + ml;
          *reinterpret_cast<float4*>(p.part_o + prow * D + d4 * 4) = acc[u];
          if (d4 == 0) reinterpret_cast<float2*>(p.part_ml)[prow] = x[u];
        }
      }
    }
  }

  // ---- fused tail: the last CTA of the unit merges the key splits; nobody waits ----
  if (up.fused_tail && p.splits > 1) {
    int32_t* counter = p.counters + unit;
    __threadfence();
    __syncthreads();
    if (tid == 0) *last_flag = (atomicAdd(counter, 1) == p.splits - 1) ? 1 : 0;
    __syncthreads();
    const bool last = *last_flag != 0;
    if (last && !*abort_flag) {
      __threadfence();
      for (int s0 = tid; s0 < M_rt * (D / 4); s0 += 4 * UM_THREADS) {
        int four[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) four[u] = s0 + u * UM_THREADS < M_rt * (D / 4) ? s0 + u * UM_THREADS : -1;
        merge_slots<D, 4, 4>(p, unit, bi, g, rt, four);
      }
    }
    // ready for the next call, whether or not this one gave up: a counter left at its final value would keep every
    // later call on this workspace from ever finding its last CTA
    if (last && tid == 0) *counter = 0;
  }

  // ---- free the tensor memory ----
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (*abort_flag) {
      drain_mmas(BAR(DRAIN));
      drain_loads(BAR(FULL_K), issued_s[0], NS);
      drain_loads(BAR(FULL_V), issued_s[1], NS);
      drain_bar(BAR(Q_FULL), 0);
    }
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------------------------------------
// Host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// 4-D bf16 tensor (D, rows, heads, batch) with element strides for the three outer axes; box = (64, box_rows, box_heads, 1),
// 128-byte swizzle, out-of-range rows read as zero.
bool make_map(CUtensorMap* m, const void* base, int D, int rows, int heads, int batch, const int64_t* stride_bhr, int box_rows,
              int box_heads) {
  EncodeTiledFn enc = encode_fn();
  if (!enc || rows < 1) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)heads, (cuuint64_t)batch};
  auto st = [&](int64_t s) { return (cuuint64_t)(s > 0 ? s * 2 : (int64_t)D * 2); };   // unused strides stay legal
  const cuuint64_t strides[3] = {st(stride_bhr[2]), st(stride_bhr[1]), st(stride_bhr[0])};
  const cuuint32_t box[4] = {64u, (cuuint32_t)box_rows, (cuuint32_t)box_heads, 1u};
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t umma_smem_bytes(int D, int KT) {
  const size_t H = D / 64;
  const size_t need = 1024 /*alignment slack*/ + 1024 /*barriers, flags*/ + H * 128 * 128 + (size_t)UM_STAGES * 2 * H * KT * 128;
  // every CTA allocates all 512 TMEM columns, so two CTAs must never share an SM: ask for more than half its shared memory
  return need > 120 * 1024 ? need : 120 * 1024;
}

template <int D>
cudaError_t launch_umma_d(const UmmaMaps& tm, const UmmaParams& up, const AttnPlan& pl, bool pdl, cudaStream_t st) {
  auto kern = attn_umma_bf16_kernel<D>;
  static SmemConfig configured;
  cudaError_t e = configure_smem(reinterpret_cast<const void*>(kern), pl.smem_bytes, configured, true);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(pl.splits, up.a.Hkv * up.row_tiles, up.a.B);
  cfg.blockDim = dim3(UM_THREADS);
  cfg.dynamicSmemBytes = pl.smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, tm, up);
}

}  // namespace

bool umma_make_map(CUtensorMap* m, const void* base, int D, int rows, int heads, int batch, const int64_t* stride_bhr, int box_rows,
                   int box_heads) {
  return make_map(m, base, D, rows, heads, batch, stride_bhr, box_rows, box_heads);
}

// Whether the tcgen05 kernel covers a shape: bf16, D in {64, 128}, block length a multiple of 16 that either keeps all
// b*G rows inside one 128-row tile or divides 128.
bool umma_supported(int dtype, int D, int M, int b) {
  if (dtype != SDLLM_BF16 || (D != 64 && D != 128) || encode_fn() == nullptr) return false;
  if (b % 16 != 0 || b > 128) return false;
  return M <= 128 || 128 % b == 0;
}

// The last CTA of a unit does the tail itself while that is a small job; otherwise a second launch spreads it over
// the whole GPU.
bool umma_tail_is_fused(const AttnPlan& pl, int D, int M) {
  // (a merge of full 128-row partials by the last CTA alone lost to the second launch at every split count measured,
  // 16.2 against 22.6 us with four splits: the last CTA does it only for small partials)
  const int forced = tuning().fused_tail;
  const bool fused = forced >= 0 ? forced == 1 : (size_t)pl.splits * (M < 128 ? M : 128) * D * 4 <= 32 * 1024;
  // the last CTA is found with a counter per unit (without an override of the splits there are never that many)
  return fused && pl.n_counters <= kWsCounters;
}

AttnPlan plan_attention_umma(int D, int M, int b, int B, int Hkv, int n1_max, const Tuning& tn) {
  AttnPlan pl{};
  pl.kind = 2; pl.cluster = 1; pl.fused_tail = true;
  pl.threads = UM_THREADS; pl.stages = UM_STAGES;
  const int sms = sm_count();
  const int G = M / b;
  pl.row_tiles = M <= 128 ? 1 : (G + 128 / b - 1) / (128 / b);
  pl.rep = M <= 32 ? 4 : (M <= 64 ? 2 : 1);
  const long long units = (long long)B * Hkv * pl.row_tiles;
  long long want = sms / units;
  if (want < 1) want = 1;
  // 8 units: sixteen splits (128 CTAs) measured 5 % ahead of eighteen (144) at every length tried
  if (want > 16 && want < 24) want = 16;
  if (tn.splits > 0) want = tn.splits;
  // Full 128-row tiles (nothing replicated): with at most 24 tiles per head eight splits beat sixteen (11.4 against 13.7 us at
  // 1024 keys, 13.1 against 14.2 at 2048). Nine splits (16 units) lost 6 % to eight wherever measured.
  if (pl.rep == 1 && tn.splits <= 0 && want > 8 && ((n1_max + 127) / 128 <= 24 || want < 16)) want = 8;
  pl.key_tile = 128;
  if (pl.rep <= 2 && (n1_max + 127) / 128 < want) pl.key_tile = 64;
  if (tn.key_tile == 64 && pl.rep <= 2) pl.key_tile = 64;
  if (tn.key_tile == 128) pl.key_tile = 128;
  pl.key_tile2 = pl.key_tile;
  const int tiles = (n1_max + pl.key_tile - 1) / pl.key_tile;
  if (want > tiles) want = tiles;
  if (want > kMaxSplits) want = kMaxSplits;
  if (want < 1) want = 1;
  pl.splits = (int)want;                // (replicas are merged inside the CTA)
  pl.part_rows = pl.splits > 1 ? (size_t)pl.row_tiles * pl.splits * (M < 128 ? M : 128) : 0;
  pl.n_counters = pl.splits > 1 ? (size_t)B * Hkv * pl.row_tiles : 0;
  pl.smem_bytes = umma_smem_bytes(D, pl.key_tile);
  return pl;
}

cudaError_t launch_attn_umma(const AttnParams& p, const AttnPlan& pl, int D, cudaStream_t st) {
  const Tuning tn = tuning();
  UmmaMaps tm;
  UmmaParams up{};
  up.a = p;
  up.a.splits = pl.splits;
  up.a.wait_cycles = tn.wait_cycles;
  up.KT = pl.key_tile; up.R = pl.rep; up.row_tiles = pl.row_tiles;
  up.heads_rt = pl.row_tiles == 1 ? p.G : 128 / p.b;
  const long long ctas = (long long)pl.splits * p.Hkv * pl.row_tiles * p.B;
  up.lpt = (p.n1_per_seq != nullptr && p.B >= 4 && p.B <= 64 && ctas > sm_count()) ? 1 : 0;
  if (tn.lpt >= 0) up.lpt = (tn.lpt == 1 && p.n1_per_seq != nullptr && p.B >= 2 && p.B <= 64) ? 1 : 0;
  up.fused_tail = umma_tail_is_fused(pl, D, p.M) ? 1 : 0;
  memset(&tm, 0, sizeof(tm));
  if (!make_map(&tm.q, p.q, D, p.b, p.Hq, p.B, p.q_stride, p.b, up.heads_rt) ||
      !make_map(&tm.k, p.k1, D, p.n1_max, p.Hkv, p.B, p.k1_stride, pl.key_tile, 1) ||
      !make_map(&tm.v, p.v1, D, p.n1_max, p.Hkv, p.B, p.k1_stride, pl.key_tile, 1))
    return cudaErrorInvalidValue;
  const bool pdl = tn.pdl != 0;
  const cudaError_t err = D == 128 ? launch_umma_d<128>(tm, up, pl, pdl, st) : launch_umma_d<64>(tm, up, pl, pdl, st);
  if (err != cudaSuccess || pl.splits == 1 || up.fused_tail || p.unfolded) return err;
  const long long merge_threads = (long long)p.B * p.Hkv * pl.row_tiles * 128 * (D / 4);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((merge_threads + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  return D == 128 ? cudaLaunchKernelEx(&cfg, umma_tail_kernel<128>, up) : cudaLaunchKernelEx(&cfg, umma_tail_kernel<64>, up);
}

// ---------------------------------------------------------------------------------------------------------
// Dispatch between the kernel families
AttnPlan plan_attention_legacy(int dtype, int D, int M, int B, int Hkv, int n_keys_max, const Tuning& tn);
cudaError_t launch_attn_legacy(const AttnParams& p, const AttnPlan& plan, int dtype, int D, cudaStream_t st);
bool kt_supported(int dtype, int D, int M, int b);
bool kt_preferred(int D, int M, int B, int Hkv, int n1_max, int n2);
AttnPlan plan_attention_kt(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn);
cudaError_t launch_attn_kt(const AttnParams& p, const AttnPlan& pl, int D, cudaStream_t st);

bool pair_supported(int dtype, int D, int M, int b);
bool plan_attention_units(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn, bool small, AttnPlan* pl);
AttnPlan plan_attention_pair(int D, int M, int b, int B, int Hkv, int n1_max, int n2, const Tuning& tn);
cudaError_t launch_attn_pair(const AttnParams& p, const AttnPlan& pl, int D, cudaStream_t st);

AttnPlan plan_attention(int dtype, int D, int M, int b, int B, int Hkv, int n1_max, int n2, bool prob_scores, bool small) {
  // bf16 goes to the tcgen05 kernels wherever they apply: heads with few query rows to the kernel that puts the keys on the
  // accumulator rows, the rest to the one that puts the queries there and has two softmax warpgroups (attn_pair.cu). fp32 and
  // the remaining bf16 shapes go to the cp.async kernels. Tuning::kernel forces a family.
  // With the probability saliency (prob_scores) the attention pass is the kernel of this file, whatever the family.
  const Tuning tn = tuning();
  if (prob_scores && tn.kernel != 1 && umma_supported(dtype, D, M, b)) return plan_attention_umma(D, M, b, B, Hkv, n1_max, tn);
  AttnPlan units;
  if (n2 > 0 && tn.kernel == 0 && umma_supported(dtype, D, 16, 16) && plan_attention_units(D, M, b, B, Hkv, n1_max, n2, tn, small, &units)) return units;
  const bool kt_ok = kt_supported(dtype, D, M, b);
  if (kt_ok && (tn.kernel == 3 || (tn.kernel == 0 && kt_preferred(D, M, B, Hkv, n1_max, n2))))
    return plan_attention_kt(D, M, b, B, Hkv, n1_max, n2, tn);
  if (tn.kernel != 1 && pair_supported(dtype, D, M, b)) return plan_attention_pair(D, M, b, B, Hkv, n1_max, n2, tn);
  AttnPlan pl = plan_attention_legacy(dtype, D, M, B, Hkv, n1_max + n2, tn);
  pl.cluster = 1; pl.warp_keys = 32; pl.kind = 0;
  pl.part_rows = pl.splits > 1 ? (size_t)pl.splits * M : 0;      // partial rows the kernels leave per (sequence, KV head)
  pl.n_counters = 0; pl.fused_tail = false;
  pl.rep = 1; pl.row_tiles = 1; pl.key_tile2 = pl.key_tile;
  return pl;
}

cudaError_t launch_attn_partial(const AttnParams& p, const AttnPlan& plan, int dtype, int D, cudaStream_t st) {
  if (plan.kind == 3) return launch_attn_kt(p, plan, D, st);
  if (plan.kind == 4) return launch_attn_pair(p, plan, D, st);
  if (plan.kind == 2) return launch_attn_umma(p, plan, D, st);
  return launch_attn_legacy(p, plan, dtype, D, st);
}

}  // namespace sdllm
