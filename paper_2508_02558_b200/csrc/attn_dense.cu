// Full-sequence bf16 attention on tcgen05 (the dense step: every row of a sequence over all of its keys).
//
// A dense contraction, bound by the tensor pipe and, in front of it, by the softmax. One CTA owns TWO 128-row query
// tiles of one query head and streams the head's K/V once for both:
//   warp 0      TMA producer: the two Q tiles, then K and V tiles (128 keys, 128-byte swizzle) into a two-slot ring
//   warp 1      tcgen05.mma issuer. Per key tile j:  S0 = Q0 K_j^T,  O1 += P1(j-1) V_(j-1),  S1 = Q1 K_j^T,
//               O0 += P0(j) V_j  -  while the softmax warps of one query tile work, the tensor pipe serves the other
//   warps 4-7   softmax of query tile 0, warps 8-11 of query tile 1: a thread owns one accumulator row (TMEM lane),
//               reads its S row, keeps the running max / sum and writes P (bf16) over S in TMEM; O accumulates in
//               TMEM and is rescaled in place only when the row's maximum grows by more than 2^8
// Tensor memory (512 columns): S0 | S1 | O0 | O1, 128 columns each (D = 64 uses half of an O region).
// The chain of one query tile is S -> softmax -> P V -> next S (P lies over S), so a key tile of a pair costs
// softmax + hand-overs + 1024 tensor cycles, with the other query tile's 1024 inside the softmax. What was taken off it
// (4540 -> 3000 cycles per pair of 128 x 128 tiles at D = 128):
//   - the MMA warp runs its loop warp-uniformly: an MMA no longer costs more to issue than to execute;
//   - P is handed over in two parts (96 keys, then 32), so that the first MMAs of P V run under the last exponentials;
//   - three-operand maxima, two-lane fp32 arithmetic, a quarter of the exponentials on the FMA pipe (poly_exp2), one
//     warp-uniform branch for the rare rescale, registers moved to the softmax warps (208 instead of 168).
// 32 heads x 1280 rows: 56.3 -> 44.0 us (34.7 with the last wave's units cut, see plan_dense); 32 (8 KV) heads x 32768 rows: 17.1 -> 14.6 ms, 1204 TFLOP/s. The long case is
// bound by power (1.6 GHz under the 1000 W cap, where a library GEMM sustains 1408); a burst at full clock runs at 1368.
// The finished rows go from TMEM through registers straight to global memory (bf16), normalised by the row sum.
// Every wait on an mbarrier is bounded; on expiry the CTA sets an abort flag, records a code in the status word and
// runs to its end (freeing its TMEM); the outputs of that call are then invalid.
#include <cuda.h>
#include <string.h>

#include "attn_device.cuh"
#include "fold.cuh"
#include "tuning.cuh"
#include "umma_host.cuh"

namespace sdllm {
using namespace dev;
namespace {

constexpr int DN_THREADS = 384;        // three warpgroups: producer and MMA issuer (and two idle warps), softmax, softmax
constexpr int DN_STAGES = 2;
constexpr int DN_POLY = 4;             // one pair of exponentials in DN_POLY is a polynomial (3 and 8 measured 1 to 2 % slower)

struct DenseMaps {
  CUtensorMap q, k, v;
};

struct DenseParams {
  const int32_t* seq_len;   // [B], nullable -> L
  void* out;                // [B, Hq, L, D] bf16 with o_stride
  float* lse;               // [B, Hq, L], nullable
  int32_t* status;          // device status word
  float* part_o;            // rows of the cut units: [unit][part][D / 4][256] float4
  float* part_ml;           // [unit][part][256] (maximum, sum)
  int B, Hq, G, L;
  int pairs;                // units of a head at full length
  int unit0, parts;         // units in front of the cut ones; CTAs that share the key tiles of a cut unit
  int second;               // cut units: 1: the launch in front is that of the same call's whole units
  float scale_log2;         // softmax scale * log2(e)
  int64_t o_stride[3];
  long long wait_cycles;    // limit of every abortable mbarrier wait
};

#include "umma_ptx.cuh"

// One query row and float4 column of a cut unit: the fold of its shares.
template <int D, int MB>
__device__ __forceinline__ void dense_fold_item(const DenseParams& p, int cut, int c4, int row) {
  constexpr int C4 = D / 4;
  const int unit = p.unit0 + cut, jp = unit % p.pairs, h = (unit / p.pairs) % p.Hq;
  const int bi = unit / (p.pairs * p.Hq);
  int n = p.seq_len ? __ldcg(p.seq_len + bi) : p.L;
  n = min(max(n, 0), p.L);
  const int r = jp * 256 + row;
  if (r >= n) return;
  const float4* po = reinterpret_cast<const float4*>(p.part_o) + ((int64_t)cut * p.parts * C4 + c4) * 256 + row;
  const float2* pm = reinterpret_cast<const float2*>(p.part_ml) + (int64_t)cut * p.parts * 256 + row;
  const FoldedColumn x = fold_splits<MB>(p.parts, [&](int s) { return __ldcg(pm + s * 256); }, [&](int s) { return __ldcg(po + (int64_t)s * C4 * 256); }, fast_exp2);
  const float inv = x.l != 0.f ? 1.f / x.l : 0.f;
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (int64_t)bi * p.o_stride[0] + (int64_t)h * p.o_stride[1] + (int64_t)r * p.o_stride[2] + c4 * 4;
  *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(x.o.x * inv, x.o.y * inv), pack_bf16(x.o.z * inv, x.o.w * inv));
  if (c4 == 0 && p.lse) p.lse[((int64_t)bi * p.Hq + h) * p.L + r] = (x.m + log2f(x.l)) * kLn2;
}
// 64 threads of whole unit `unit` (which have 72 registers each) fold their part of all cut units, 64 rows of one column at a time.
template <int D>
__device__ __forceinline__ void dense_fold_share(const DenseParams& p, int unit, int thread) {
  const int tasks = (p.pairs * p.Hq * p.B - p.unit0) * (D / 4) * 4;
  for (int t = unit; t < tasks; t += p.unit0) dense_fold_item<D, 6>(p, t / D, t / 4 % (D / 4), (t & 3) * 64 + thread);
}

// MODE (variants of their own: the plain one has no register to spare):
//   DN_CUT     the CTA takes a share of a unit's key tiles
//   DN_BEHIND  the launch in front is that of the same call's cut units: it is not waited for at the start, and two idle warps wait
//              for it to fold what it leaves
constexpr int DN_PLAIN = 0, DN_CUT = 1, DN_BEHIND = 2;
template <int D, int MODE>
__global__ void __launch_bounds__(DN_THREADS, 1) dense_attn_bf16_kernel(const __grid_constant__ DenseMaps tm, const DenseParams p) {
  constexpr bool CUT = MODE == DN_CUT;
  extern __shared__ unsigned char smem_raw[];
  constexpr int H = D / 64;                 // 64-column halves of a row (128 bytes each: one swizzle atom wide)
  constexpr int KT = 128;                   // keys per tile
  constexpr int NS = DN_STAGES;
  constexpr int HALF = KT * 128;            // bytes of one 64-column half of a 128-row tile
  constexpr int TILE = H * HALF;            // bytes of a Q, K or V tile
  constexpr uint32_t S_COL0 = 0, O_COL0 = 256, T_STRIDE = 128;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // (the plain variant takes its place from the grid as it is: values that the compiler knows to be warp-uniform, sequence length
  // and loop bounds included, stay in uniform registers; from a linear index it ran 2.5 % slower)
  const int part = CUT ? blockIdx.x % (unsigned)p.parts : 0, unit = CUT ? p.unit0 + (int)(blockIdx.x / (unsigned)p.parts) : 0;
  const int jp = CUT ? unit % p.pairs : blockIdx.x, h = CUT ? (unit / p.pairs) % p.Hq : blockIdx.y, g = h / p.G;
  const int bi = CUT ? unit / (p.pairs * p.Hq) : blockIdx.z;

  if (!CUT && (bi * p.Hq + h) * p.pairs + jp >= p.unit0) {   // one of the units that are cut
    if (MODE == DN_BEHIND) grid_dependency_wait();
    return;
  }
  if (MODE != DN_BEHIND && (!CUT || !p.second)) grid_dependency_wait();    // everything this kernel reads may come from the kernel in front of it
  grid_launch_dependents();
  int n = p.seq_len ? p.seq_len[bi] : p.L;
  n = min(max(n, 0), p.L);
  const int row00 = 2 * jp * 128;           // first row of query tile 0; query tile 1 starts 128 rows further
  if (row00 >= n) {                         // both query tiles lie past the sequence's end (whole CTA, before any set-up)
    if (CUT && p.second) grid_dependency_wait();
    if (MODE == DN_BEHIND) {
      grid_dependency_wait();
      if (tid < 64) dense_fold_share<D>(p, (bi * p.Hq + h) * p.pairs + jp, tid);
    }
    return;
  }
  const bool act1 = row00 + 128 < n;
  const int nt_all = (n + KT - 1) / KT;     // key tiles of the unit; this CTA takes [t0, t0 + nt)
  const int t0 = CUT ? part * nt_all / p.parts : 0, nt = CUT ? (part + 1) * nt_all / p.parts - t0 : nt_all;

  const uint32_t raw_addr = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t bars = smem_u32(smem);
  auto BAR = [&](int i) { return bars + 8u * (uint32_t)i; };
  const int Q_FULL = 0, FULL_K = 1, FULL_V = 1 + NS, EMPTY_K = 1 + 2 * NS, EMPTY_V = 1 + 3 * NS;
  const int S_FULL = 1 + 4 * NS, P_FULL = S_FULL + 2, PV_DONE = S_FULL + 6, DRAIN = S_FULL + 8;   // P_FULL: two parts per query tile
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 260);
  int* issued_s = reinterpret_cast<int*>(smem + 264);        // [2] tiles whose K / V loads are on their way (for an aborted CTA's way out)
  unsigned char* q_s = smem + 1024;
  unsigned char* stage0 = q_s + 2 * TILE;

  if (tid == 0) {
    prefetch_tmap(&tm.q); prefetch_tmap(&tm.k); prefetch_tmap(&tm.v);
    mbar_init(BAR(Q_FULL), 1);
    for (int i = 0; i < NS; ++i) {
      mbar_init(BAR(FULL_K + i), 1); mbar_init(BAR(FULL_V + i), 1);
      mbar_init(BAR(EMPTY_K + i), 1); mbar_init(BAR(EMPTY_V + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(S_FULL + i), 1);
      mbar_init(BAR(P_FULL + 2 * i), 4);   // the four softmax warps of a query tile
      mbar_init(BAR(P_FULL + 2 * i + 1), 4);
      mbar_init(BAR(PV_DONE + i), 1);
    }
    mbar_init(BAR(DRAIN), 1);
    *abort_flag = 0;
    issued_s[0] = issued_s[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {                          // the MMA warp owns the tensor memory
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  auto tile_nv = [&](int j) { return min(n - (t0 + j) * KT, KT); };     // valid keys of this CTA's tile j (> 0 for j < nt)

  // Registers move from the first warpgroup to the softmax warps: 128 * (72 + 2 * 208) of the 384 * 168 at launch.
  if (warp < 4) {
    regs_dec_72();
    if (warp == 0) {
      // ======================================= TMA producer =======================================
      if (lane == 0 && (!CUT || nt > 0)) {
        mbar_expect_tx(BAR(Q_FULL), (uint32_t)((act1 ? 2 : 1) * TILE));
        for (int t = 0; t < (act1 ? 2 : 1); ++t)
          for (int hh = 0; hh < H; ++hh)
            tma_load_4d(smem_u32(q_s + t * TILE + hh * HALF), &tm.q, BAR(Q_FULL), hh * 64, row00 + t * 128, h, bi);
        int k_issued = 0, v_issued = 0;
        for (int j = 0; j < nt; ++j) {
          const int s = j % NS;
          const uint32_t ph = ((j / NS) - 1) & 1;
          const uint32_t kdst = smem_u32(stage0 + (size_t)s * 2 * TILE), vdst = kdst + TILE;
          if (j >= NS && !wait_bar(BAR(EMPTY_K + s), ph, abort_flag, p.status, 21, p.wait_cycles)) break;
          mbar_expect_tx(BAR(FULL_K + s), (uint32_t)TILE);
          for (int hh = 0; hh < H; ++hh) tma_load_4d(kdst + hh * HALF, &tm.k, BAR(FULL_K + s), hh * 64, (t0 + j) * KT, g, bi);
          k_issued = j + 1;
          if (j >= NS && !wait_bar(BAR(EMPTY_V + s), ph, abort_flag, p.status, 22, p.wait_cycles)) break;
          mbar_expect_tx(BAR(FULL_V + s), (uint32_t)TILE);
          for (int hh = 0; hh < H; ++hh) tma_load_4d(vdst + hh * HALF, &tm.v, BAR(FULL_V + s), hh * 64, (t0 + j) * KT, g, bi);
          v_issued = j + 1;
        }
        issued_s[0] = k_issued; issued_s[1] = v_issued;
      }
    } else if (warp == 1) {
      // ======================================= MMA issuer =======================================
      // The whole warp walks the tiles and one elected lane issues: with everything around the MMAs warp-uniform their
      // descriptors live in uniform registers and an MMA costs a few instructions. (A loop run by one lane alone took about
      // 600 cycles to issue eight MMAs, more than their 512 cycles of execution.)
      const bool leader = elect_one();
      const uint32_t idesc_pv = instr_desc(D, true);
      const uint64_t q_desc = smem_desc(smem_u32(q_s), 16u, 1024u), k_desc = smem_desc(smem_u32(stage0), 16u, 1024u);
      const uint64_t v_desc = smem_desc(smem_u32(stage0) + TILE, (uint32_t)HALF, 1024u);
      bool ok = (!CUT || nt > 0) && wait_bar_warp(BAR(Q_FULL), 0, abort_flag, p.status, 23, p.wait_cycles);
      // S_t = Q_t K_j^T into the S region of query tile t
      auto issue_s = [&](int t, int j) {
        const uint32_t idesc_s = instr_desc((tile_nv(j) + 15) & ~15, false);
        const uint32_t d_t = tmem_base + S_COL0 + (uint32_t)t * T_STRIDE;
        const uint64_t qd = q_desc + (uint64_t)(t * (TILE >> 4)), kd = k_desc + (uint64_t)((j % NS) * (2 * TILE >> 4));
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint64_t off = (uint64_t)(((ks >> 2) * HALF + (ks & 3) * 32) >> 4);
            mma_ss(d_t, qd + off, kd + off, idesc_s, ks > 0 ? 1u : 0u);
          }
          tc_commit(BAR(S_FULL + t));
        }
        __syncwarp();
      };
      // O_t += P_t V_j as the softmax warps of query tile t hand P_t over; `release` frees the V slot afterwards
      auto issue_pv = [&](int t, int j, bool release) -> bool {
        const int s = j % NS;
        if (!wait_bar_warp(BAR(FULL_V + s), (j / NS) & 1, abort_flag, p.status, 25, p.wait_cycles)) return false;
        const uint64_t vd = v_desc + (uint64_t)(s * (2 * TILE >> 4));
        const uint32_t a_t = tmem_base + S_COL0 + (uint32_t)t * T_STRIDE, o_t = tmem_base + O_COL0 + (uint32_t)t * T_STRIDE;
        const int n_ks = (tile_nv(j) + 15) >> 4;
#pragma unroll
        for (int part = 0; part < 2; ++part) {          // the first 96 keys start while P of the other 32 is still being made
          if (!wait_bar_warp(BAR(P_FULL + 2 * t + part), j & 1, abort_flag, p.status, 24, p.wait_cycles)) return false;
          tc_fence_after();
          if (leader) {
#pragma unroll
            for (int ks = part * 6; ks < 6 + 2 * part; ++ks)
              if (ks < n_ks) mma_ts(o_t, a_t + ks * 8, vd + ks * (2048 >> 4), idesc_pv, (j > 0 || ks > 0) ? 1u : 0u);
          }
        }
        if (leader) {
          tc_commit(BAR(PV_DONE + t));
          if (release) tc_commit(BAR(EMPTY_V + s));
        }
        __syncwarp();
        return true;
      };
      ok = ok && wait_bar_warp(BAR(FULL_K), 0, abort_flag, p.status, 26, p.wait_cycles);
      for (int j = 0; j < nt && ok; ++j) {
        const int s = j % NS;
        tc_fence_after();
        issue_s(0, j);
        if (act1) {
          if (j > 0 && !issue_pv(1, j - 1, true)) { ok = false; break; }
          issue_s(1, j);
        }
        if (leader) tc_commit(BAR(EMPTY_K + s));
        // (the next K tile is waited for here, ahead of P: nothing then stands between this P V and the next S)
        if (j + 1 < nt && !wait_bar_warp(BAR(FULL_K + (j + 1) % NS), ((j + 1) / NS) & 1, abort_flag, p.status, 26, p.wait_cycles)) { ok = false; break; }
        if (!issue_pv(0, j, !act1)) { ok = false; break; }
      }
      if (ok && act1) ok = issue_pv(1, nt - 1, true);
    } else if (MODE == DN_BEHIND) {
      // ======================================= fold of the cut units =======================================
      grid_dependency_wait();
      dense_fold_share<D>(p, (bi * p.Hq + h) * p.pairs + jp, tid - 64);
    }
  } else {
    // ======================================= softmax warps =======================================
    regs_inc_208();
    const int t = (warp - 4) >> 2;                     // query tile of this warp
    const int q4 = warp & 3;                           // TMEM lane quadrant this warp may access
    const int row = q4 * 32 + lane;
    if (t == 0 || act1) {
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
      const uint32_t s_addr = lane_addr + S_COL0 + (uint32_t)t * T_STRIDE;
      const uint32_t o_addr = lane_addr + O_COL0 + (uint32_t)t * T_STRIDE;
      float m_run = -INFINITY, l_run = 0.f;
      bool ok = true;
      for (int j = 0; j < nt && ok; ++j) {
        const int nv = tile_nv(j);
        if (!wait_bar_warp(BAR(S_FULL + t), j & 1, abort_flag, p.status, 27, p.wait_cycles)) { ok = false; break; }
        tc_fence_after();
        uint32_t sv[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, sv[c]);
        tc_wait_ld();
        if (nv < KT) {                                   // the ragged last tile: keys past the end count as -inf
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c * 32 + i >= nv) sv[c][i] = __float_as_uint(-INFINITY);
        }
        float m8[8];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float a = __uint_as_float(sv[c][2 * i]), b = __uint_as_float(sv[c][2 * i + 1]);
            m8[i & 7] = c == 0 && i < 8 ? fmaxf(a, b) : max3(m8[i & 7], a, b);
          }
        const float mx = max3(max3(m8[0], m8[1], m8[2]), max3(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7]));
        // running maximum: O (in TMEM) and l are rescaled only when the maximum grows by more than 2^8
        const float m_new = fmaxf(m_run, mx * p.scale_log2);
        const bool grow = m_new > m_run + 8.f;          // also true on the first finite maximum
        if (__any_sync(0xffffffffu, grow)) {
          const float alpha = grow ? fast_exp2(m_run - m_new) : 1.f;      // 0 when m_run is -inf
          if (grow) m_run = m_new == INFINITY ? NAN : m_new;       // a logit of +inf: the row is NaN from here on
          l_run = l_run < kNanSum ? l_run * alpha : NAN;
          if (j > 0) {
            // every PV of this query tile issued so far must have landed before its rows are rewritten
            if (!wait_bar_warp(BAR(PV_DONE + t), (j - 1) & 1, abort_flag, p.status, 28, p.wait_cycles)) { ok = false; break; }
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
              uint32_t ov[16];
              tmem_ld16(o_addr + c * 16, ov);
              tc_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
              tmem_st16(o_addr + c * 16, ov);
            }
          }
        }
        const float mu = (m_run == -INFINITY) ? 0.f : m_run;
        // V rows past the sequence's end may hold anything: query tile 0 zeroes them so that 0 * V stays 0
        const int n_mma = (nv + 15) & ~15;
        if (t == 0 && nv < n_mma) {
          const int s = j % NS;
          if (!wait_bar_warp(BAR(FULL_V + s), (j / NS) & 1, abort_flag, p.status, 29, p.wait_cycles)) { tc_wait_st(); ok = false; break; }   // (stores to tensor memory may be under way)
          unsigned char* vs = stage0 + (size_t)s * 2 * TILE + TILE;
          const int nz = (n_mma - nv) * H * 8;           // 16-byte chunks to clear
          for (int i = q4 * 32 + lane; i < nz; i += 128) {
            const int rr = nv + i / (H * 8), c = i % (H * 8);
            *reinterpret_cast<uint4*>(vs + (c >> 3) * HALF + rr * 128 + (((c & 7) ^ (rr & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async();
        }
        // P = exp2(S * scale_log2 - mu) as bf16 over the first 64 columns of the S region, handed over in two parts
        const uint64_t scale2 = pack_f2(p.scale_log2, p.scale_log2), mu2 = pack_f2(-mu, -mu);
        uint64_t ps[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float x0, x1, e0, e1;
            unpack_f2(fma_f2(pack_f2(__uint_as_float(sv[c][2 * i]), __uint_as_float(sv[c][2 * i + 1])), scale2, mu2), x0, x1);
            if (i % DN_POLY == DN_POLY - 1) {
              poly_exp2(x0, x1, e0, e1);
            } else {
              e0 = fast_exp2(x0);
              e1 = fast_exp2(x1);
            }
            ps[i & 3] = add_f2(ps[i & 3], pack_f2(e0, e1));
            pk[i] = pack_bf16(e0, e1);
          }
          tmem_st16(s_addr + c * 16, pk);
          if (c >= 2) {
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR(P_FULL + 2 * t + (c - 2)));
          }
        }
        {
          float a, b;
          unpack_f2(add_f2(add_f2(ps[0], ps[1]), add_f2(ps[2], ps[3])), a, b);
          l_run += a + b;
        }
      }
      // ---- the finished row: TMEM -> registers -> normalise -> bf16 -> global memory ----
      if (ok) ok = (!CUT || nt > 0) && wait_bar_warp(BAR(PV_DONE + t), (nt - 1) & 1, abort_flag, p.status, 30, p.wait_cycles);
      tc_fence_after();
      const int r_glob = row00 + t * 128 + row;
      // (written behind the wait: ahead of it, two selects on l_run cost the loop above 3 %)
      const float l_fin = l_run >= kNanSum ? NAN : (m_run == -INFINITY && l_run < 1.f ? 0.f : l_run);   // 0: only logits of -inf, which poly_exp2 does not make 0
      if constexpr (CUT) {
        // A share of a unit: un-normalised rows and their (maximum, sum) go to the workspace, float4 columns apart so that the
        // lanes of a warp write in a row; dense_fold_kernel folds them.
        const int64_t slot = blockIdx.x;
        float4* po = reinterpret_cast<float4*>(p.part_o) + slot * (D / 4) * 256 + t * 128 + row;
        if (ok) {
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {
            uint32_t ov[16];
            tmem_ld16(o_addr + c * 16, ov);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 4; ++i)
              __stcg(po + (c * 4 + i) * 256, make_float4(__uint_as_float(ov[4 * i]), __uint_as_float(ov[4 * i + 1]), __uint_as_float(ov[4 * i + 2]),
                                                         __uint_as_float(ov[4 * i + 3])));
          }
        }
        __stcg(reinterpret_cast<float2*>(p.part_ml) + slot * 256 + t * 128 + row, make_float2(m_run, ok ? l_fin : 0.f));
      } else if (ok) {
        const float inv = l_fin != 0.f ? 1.f / l_fin : 0.f;
        __nv_bfloat16* orow = reinterpret_cast<__nv_bfloat16*>(p.out) + (int64_t)bi * p.o_stride[0] + (int64_t)h * p.o_stride[1] +
                              (int64_t)r_glob * p.o_stride[2];
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t ov[32];
          tmem_ld32(o_addr + c * 32, ov);               // warp-wide: every lane takes part, valid row or not
          tc_wait_ld();
          if (r_glob < n) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint4 w4;
              w4.x = pack_bf16(__uint_as_float(ov[8 * i]) * inv, __uint_as_float(ov[8 * i + 1]) * inv);
              w4.y = pack_bf16(__uint_as_float(ov[8 * i + 2]) * inv, __uint_as_float(ov[8 * i + 3]) * inv);
              w4.z = pack_bf16(__uint_as_float(ov[8 * i + 4]) * inv, __uint_as_float(ov[8 * i + 5]) * inv);
              w4.w = pack_bf16(__uint_as_float(ov[8 * i + 6]) * inv, __uint_as_float(ov[8 * i + 7]) * inv);
              *reinterpret_cast<uint4*>(orow + c * 32 + i * 8) = w4;
            }
          }
        }
        if (r_glob < n && p.lse) p.lse[((int64_t)bi * p.Hq + h) * p.L + r_glob] = (m_run + log2f(l_fin)) * kLn2;
      }
    }
  }

  // ---- teardown ----
  if (CUT && p.second) grid_dependency_wait();      // this launch must not be over before the one in front of it is
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    if (__builtin_expect(*abort_flag, 0)) {
      if (lane == 0) {
        drain_loads(BAR(FULL_K), issued_s[0], NS);
        drain_loads(BAR(FULL_V), issued_s[1], NS);
        if (issued_s[0] > 0) drain_bar(BAR(Q_FULL), 0);
      }
    }
  }
  if (warp == 1) {
    if (__builtin_expect(*abort_flag, 0)) drain_mmas(BAR(DRAIN));
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

size_t dense_smem_bytes(int D) {
  const size_t tile = (size_t)(D / 64) * 128 * 128;
  return 1024 /*alignment slack*/ + 1024 /*barriers*/ + 2 * tile + (size_t)DN_STAGES * 2 * tile;
}

// Fold of the shares of the cut units: one thread per query row and float4 column, lanes along the rows.
template <int D>
__global__ void __launch_bounds__(256) dense_fold_kernel(const DenseParams p) {
  grid_dependency_wait();
  grid_launch_dependents();
  dense_fold_item<D, 8>(p, blockIdx.x / (D / 4), blockIdx.x % (D / 4), threadIdx.x);
}

// How the units (a sequence's head and pair of query tiles) of a call are launched: the first `whole` of them one CTA each, the
// rest - what the last full wave leaves over, or all of less than a wave - with their key tiles shared out to `parts` CTAs. A
// unit takes a whole SM, so without that 160 units on 148 SMs run in two waves (32 heads x 1280 rows: 44.0 us).
// Costs in us beyond the full waves: a key tile 1.55, a CTA's set-up and way out 6.5.
//   front   the cut units' launch first; the whole ones take the SMs as they come free and two idle warps of each fold the partial
//           rows: 2 more for the partial rows and 0.25 per share (32 heads x 1280: 34.7 us; 8 x 5000: 90). A task of the fold, 64 rows
//           of one float4 column, takes those warps 1.1 per six shares, up to 0.6 of a CTA's time. Per wave the whole units' variant is 2 %
//           slower and the fold costs a tenth of its time there (head dimension 64, whose softmax is short of issue slots: 7 % from the second wave
//           on, and three tenths), so this is for few cut units and few waves. 110 calls of one wave to six, behind / in front wherever the fold fits / by this rule: 16 heads x 5402, 56 cut
//           units, 207.6 / 231.5 / 207.4; 32 x 2618 of head dimension 64, 56 cut units, 104.6 / 117.2 / 102.7; 64 x 1240, 24 cut, 65.0 / 60.8 / 60.8.
//   behind  the cut units' launch overlaps the last wave and 2 of its set-up, a launch of its own folds: 7.25 (3 of it a margin)
//           and 0.35 per share (40.4 and 94.4 us; 32 heads x 2600, 56 cut units: 116, and 124 with them in front).
// Batches of several sequences may be ragged, which the host cannot see: they are cut only where all units fit one wave.
struct DensePlan {
  int whole, parts;
  bool front;
};
DensePlan plan_dense(int B, int Hq, int L, int D) {
  const int sms = sm_count(), nt = (L + 127) / 128, pairs = (nt + 1) / 2;
  const long long units = (long long)B * Hq * pairs, rest = units % sms;
  DensePlan pl{(int)units, 1, false};
  if (rest == 0 || (B > 1 && rest != units)) return pl;
  const double whole = 6.5 + 1.55 * nt;
  double least = whole;
  for (int q = 2; q <= 16 && q <= nt && rest * q <= sms; ++q) {
    const double tiles = 1.55 * ((nt + q - 1) / q), behind = (rest == units ? 6.5 : 4.5) + tiles + 7.25 + 0.35 * q;
    const double fold = 1.1 * ((q + 5) / 6) * (double)(rest * D) / (double)(units - rest), waves = (double)((units - rest) / sms);
    const double in_front = 8.5 + tiles + 0.25 * q + (D == 64 ? 0.07 * whole * (waves - 1) + 0.3 * fold * waves : (0.02 * whole + 0.1 * fold) * waves);
    const bool front = rest != units && fold <= 0.6 * whole && in_front < behind;
    const double cost = front ? in_front : behind;
    if (cost < least) { least = cost; pl.whole = (int)(units - rest); pl.parts = q; pl.front = front; }
  }
  return pl;
}

cudaError_t launch_overlapped(const void* kern, void** args, dim3 grid, int threads, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = tuning().pdl != 0 ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, kern, args);
}

template <int D>
cudaError_t launch_dense_d(const DenseMaps& tm, DenseParams p, const DensePlan& pl, int units, cudaStream_t st) {
  const void *kern = pl.front ? reinterpret_cast<const void*>(dense_attn_bf16_kernel<D, DN_BEHIND>) : reinterpret_cast<const void*>(dense_attn_bf16_kernel<D, DN_PLAIN>),
             *cut_kern = reinterpret_cast<const void*>(dense_attn_bf16_kernel<D, DN_CUT>);
  static SmemConfig plain_configured, behind_configured, cut_configured;
  const size_t smem = dense_smem_bytes(D);
  cudaError_t e = configure_smem(kern, smem, pl.front ? behind_configured : plain_configured, true);
  if (e == cudaSuccess) e = configure_smem(cut_kern, smem, cut_configured, true);
  if (e != cudaSuccess) return e;
  void* args[2] = {const_cast<DenseMaps*>(&tm), &p};
  p.parts = pl.parts; p.unit0 = pl.whole; p.second = 0;
  const dim3 whole_grid(p.pairs, p.Hq, p.B), cut_grid((unsigned)((units - pl.whole) * pl.parts));
  // The second launch of a call need not wait for the first (it depends on what that one depends on, and every CTA of the first has
  // seen that complete before it lets the next launch start), so its CTAs take the SMs that are idle; each waits for the first launch
  // before its own end, so that nothing behind them starts before both are done.
  if (pl.front) {
    e = launch_overlapped(cut_kern, args, cut_grid, DN_THREADS, smem, st);
    return e != cudaSuccess ? e : launch_overlapped(kern, args, whole_grid, DN_THREADS, smem, st);
  }
  if (pl.whole > 0) {
    e = launch_overlapped(kern, args, whole_grid, DN_THREADS, smem, st);
    if (e != cudaSuccess || pl.whole == units) return e;
    p.second = tuning().pdl != 0 ? 1 : 0;
  }
  e = launch_overlapped(cut_kern, args, cut_grid, DN_THREADS, smem, st);
  if (e != cudaSuccess) return e;
  void* fold_args[1] = {&p};
  return launch_overlapped(reinterpret_cast<const void*>(dense_fold_kernel<D>), fold_args, dim3((unsigned)((units - pl.whole) * (D / 4))), 256, 0, st);
}

}  // namespace

int dense_launches(int B, int Hq, int L, int D) {
  const DensePlan pl = plan_dense(B, Hq, L, D);
  return pl.parts == 1 ? 1 : (pl.whole > 0 && !pl.front ? 3 : 2);
}

DenseWorkspace dense_workspace(int B, int Hq, int L, int D) {
  const DensePlan pl = plan_dense(B, Hq, L, D);
  const long long units = (long long)B * Hq * ((L + 255) / 256);
  const size_t rows = pl.parts > 1 ? (size_t)(units - pl.whole) * pl.parts * 256 : 0;
  DenseWorkspace w{};
  w.part_o = kWsDataOffset;
  w.part_ml = w.part_o + rows * D * 4;
  w.total = rows > 0 ? w.part_ml + rows * 2 * 4 : kWsStatusBytes;
  return w;
}

cudaError_t launch_dense(const DenseCall& c, cudaStream_t st) {
  const int pairs = (c.L + 255) / 256;
  const long long units = (long long)c.B * c.Hq * pairs;
  if (c.Hq > 65535 || c.B > 65535 || units > 0x7fffffffLL / 16) return cudaErrorInvalidValue;
  DenseMaps tm;
  memset(&tm, 0, sizeof(tm));
  bool ok = umma_make_map(&tm.q, c.q, c.D, c.L, c.Hq, c.B, c.q_stride, 128, 1);
  ok = ok && umma_make_map(&tm.k, c.k, c.D, c.L, c.Hkv, c.B, c.kv_stride, 128, 1);
  ok = ok && umma_make_map(&tm.v, c.v, c.D, c.L, c.Hkv, c.B, c.kv_stride, 128, 1);
  if (!ok) return cudaErrorInvalidValue;
  DensePlan pl = plan_dense(c.B, c.Hq, c.L, c.D);
  const DenseWorkspace w = dense_workspace(c.B, c.Hq, c.L, c.D);
  if (c.workspace_bytes < w.total) pl = {(int)units, 1, false};
  DenseParams p{};
  p.seq_len = c.seq_len; p.out = c.out; p.lse = c.lse; p.status = reinterpret_cast<int32_t*>(c.workspace);
  p.part_o = reinterpret_cast<float*>(reinterpret_cast<char*>(c.workspace) + w.part_o);
  p.part_ml = reinterpret_cast<float*>(reinterpret_cast<char*>(c.workspace) + w.part_ml);
  p.B = c.B; p.Hq = c.Hq; p.G = c.Hq / c.Hkv; p.L = c.L; p.pairs = pairs;
  p.scale_log2 = c.scale * kLog2e;
  p.wait_cycles = tuning().wait_cycles;
  for (int i = 0; i < 3; ++i) p.o_stride[i] = c.o_stride[i];
  return c.D == 128 ? launch_dense_d<128>(tm, p, pl, (int)units, st) : launch_dense_d<64>(tm, p, pl, (int)units, st);
}

}  // namespace sdllm
