// Selection of the kept entries, pooling, the row gather and the fold of key splits as device functions, shared by the kernels that
// select (select_compact.cu, refresh_select.cu). Included inside namespace sdllm { namespace { ... } } of each of them.
#pragma once

#include "umma_ptx.cuh"

// Order-preserving map fp32 -> u32 (larger float <=> larger key). -0 is folded onto +0 and NaN sorts lowest so the
// order agrees with a numeric comparison of the values. No value maps to 0, which stands for "no candidate".
__device__ __forceinline__ uint32_t score_key(float x) {
  if (x != x) return 1u;
  if (x == 0.f) x = 0.f;
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---------------------------------------------------------------------------------------------------------
// Selection of one (sequence, KV head).
//
// A head's candidates are a few kilobytes of scores, so the selection is a chain of latencies: what counts is the number of
// barriers on it and the instructions that stand in each other's way. SW warps select; each owns a contiguous run of
// candidates, held in registers (item j of a thread is candidate c0 + 32 j of its warp's run, so warp order, item order,
// lane order is position order). A radix pass (four of 8 bits, most significant first) is one histogram by shared-memory
// atomics and ONE barrier of the selecting warps: the histograms of all passes are cleared before the scores are waited
// for, and each warp scans the 256 bins itself instead of waiting for one of them to publish the decision. With all 32
// warps of a CTA doing that the scan is bound by instruction issue (1650 cycles per pass, and 560 more per candidate and
// thread where lanes with equal bins were first counted by match.any); with 8 warps and plain atomics a pass takes 890.
// The ordered emission takes a key's rank from ballots and the warps' totals, with one more barrier. (Selection and gather
// of 32 heads x 1248 candidates: 9.9 -> 8.4 us; six of its seven phases are now about 0.5 us each.) Counts are integers,
// so nothing depends on the order in which threads or atomics run: the result is deterministic.
//
// CS > 1: the CTAs of a thread-block cluster share the head, each holding a contiguous slice. A CTA adds its histogram of a
// pass into every peer's with remote shared-memory atomics, and a cluster barrier takes the place of the CTA's.
struct HeadPlace {
  int C, o, b;                 // candidates, block offset, block length: candidate c sits at position c < o ? c : c + b
  int n0, n1;                  // entries kept from the first / second segment
  int c1;                      // the segments are [0, c1) and [c1, C)
  int kept;                    // n0 + n1
};

__device__ __forceinline__ HeadPlace place_head(const SelectParams& p, int L, int o) {
  HeadPlace h;
  L = min(max(L, 0), p.Lmax);
  h.b = p.b;
  h.o = min(max(o, 0), max(L - p.b, 0));
  h.C = max(L - p.b, 0);
  int n_pre, n_suf;
  const int n_total = keep_count_total(h.o, h.C - h.o, p.retention, p.mode, &n_pre, &n_suf);
  if (p.mode == SDLLM_SELECT_JOINT_FLOOR) {
    h.c1 = h.C;
    h.n0 = min(n_total, p.n_keep_max);
    h.n1 = 0;
  } else {
    h.c1 = h.o;
    h.n0 = min(n_pre, p.n_keep_max);
    h.n1 = min(n_suf, p.n_keep_max - h.n0);
  }
  h.kept = h.n0 + h.n1;        // (a quota never exceeds its segment)
  return h;
}

template <int SW, int CS>
struct SelectShared {
  uint32_t hist[2][4][256];                        // one per segment and radix pass
  uint32_t sum[CS > 1 ? 2 : 1][CS > 1 ? 4 : 1][CS > 1 ? 256 : 1];   // the cluster's histograms
  uint32_t tot_gt[2][SW], tot_eq[2][SW];           // survivors and ties of a warp
  uint32_t cta_gt[2][CS], cta_eq[2][CS];           // ... and of the cluster's CTAs
  // what has to be zero before a selection starts
  __device__ __forceinline__ void clear(int tid, int nt) {
    for (int i = tid; i < (int)(sizeof(hist) / 16); i += nt) reinterpret_cast<uint4*>(&hist[0][0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (CS > 1)
      for (int i = tid; i < (int)(sizeof(sum) / 16); i += nt) reinterpret_cast<uint4*>(&sum[0][0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  }
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// Address, in the shared memory of CTA `rank` of the cluster, of the word that lives at `local` in this CTA's.
__device__ __forceinline__ uint32_t peer_address(const uint32_t* local, uint32_t rank) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(ra) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  return ra;
}
__device__ __forceinline__ void peer_add(uint32_t address, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;\n" ::"r"(address), "r"(v) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t address, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(address), "r"(v) : "memory");
}
template <int SW>
__device__ __forceinline__ void select_barrier() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(32 * SW) : "memory");
}

// The threads of the SW selecting warps call this with their keys (item j is candidate c0 + 32 j; key 0: none).
// emit(w, c) is called for every kept candidate c with its rank w in the head's ascending list.
template <int SW, int KPT, int CS, typename Emit>
__device__ __forceinline__ void select_head(const HeadPlace& h, const uint32_t (&key)[KPT], int c0, SelectShared<SW, CS>& sh, int rank, Emit emit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t run_out = 0;                                // entries of the segment before
#pragma unroll 1
  for (int si = 0; si < 2; ++si) {
    const int c_lo = si == 0 ? 0 : h.c1, c_hi = si == 0 ? h.c1 : h.C, n = si == 0 ? h.n0 : h.n1;
    if (n <= 0 || c_hi <= c_lo) continue;              // (the same decision in every CTA of a cluster)
    uint32_t in = 0u;                                  // items with a candidate of the segment
#pragma unroll
    for (int j = 0; j < KPT; ++j) in |= key[j] != 0u && c0 + 32 * j >= c_lo && c0 + 32 * j < c_hi ? 1u << j : 0u;
    uint32_t thr = 0u, need_eq = 0u;                   // (as they stand: everything is kept)
    if (n < c_hi - c_lo) {
      uint32_t remaining = (uint32_t)n;
#pragma unroll 1
      for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const uint32_t himask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
        uint32_t* hist = sh.hist[si][pass];
#pragma unroll
        for (int j = 0; j < KPT; ++j)
          if ((in >> j & 1u) != 0u && (key[j] & himask) == thr) atomicAdd(&hist[(key[j] >> shift) & 0xFFu], 1u);
        if constexpr (CS > 1) {
          __syncthreads();
          for (int i = tid; i < 256 * CS; i += 32 * SW) {
            const uint32_t v = hist[i & 255];
            if (v != 0u) peer_add(peer_address(&sh.sum[si][pass][i & 255], (uint32_t)(i >> 8)), v);
          }
          cluster_barrier();
          hist = sh.sum[si][pass];
        } else {
          select_barrier<SW>();
        }
        // lane handles bins [255 - 8*lane - 7, 255 - 8*lane], scanning downward; every warp takes the same decision
        const uint4 lo = *reinterpret_cast<const uint4*>(&hist[248 - 8 * lane]), hi = *reinterpret_cast<const uint4*>(&hist[252 - 8 * lane]);
        const uint32_t local[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += local[i];
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += y;
        }
        const int src = __ffs(__ballot_sync(0xffffffffu, incl >= remaining)) - 1;
        uint32_t above = incl - sum;                   // candidates in bins above this lane's range
        uint32_t bin = 0, left = remaining;
        bool found = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (!found && above + local[i] >= remaining) { found = true; bin = 255u - (8u * lane + i); left = remaining - above; }
          above += local[i];
        }
        thr |= __shfl_sync(0xffffffffu, bin, src) << shift;
        remaining = __shfl_sync(0xffffffffu, left, src);
      }
      need_eq = remaining;                             // how many candidates equal to thr are still to be kept (>= 1)
    }
    // ---- ordered emission ----
    uint32_t n_gt = 0, n_eq = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      n_gt += (in >> j & 1u) != 0u && key[j] > thr ? 1u : 0u;
      n_eq += (in >> j & 1u) != 0u && key[j] == thr ? 1u : 0u;
    }
    n_gt = __reduce_add_sync(0xffffffffu, n_gt);
    n_eq = __reduce_add_sync(0xffffffffu, n_eq);
    if (lane == 0) { sh.tot_gt[si][warp] = n_gt; sh.tot_eq[si][warp] = n_eq; }
    if constexpr (CS > 1) __syncthreads(); else select_barrier<SW>();
    const uint32_t gt_all = lane < SW ? sh.tot_gt[si][lane] : 0u, eq_all = lane < SW ? sh.tot_eq[si][lane] : 0u;
    uint32_t gt_before = __reduce_add_sync(0xffffffffu, lane < warp ? gt_all : 0u);
    uint32_t eq_before = __reduce_add_sync(0xffffffffu, lane < warp ? eq_all : 0u);
    if constexpr (CS > 1) {
      if (warp == 0) {
        const uint32_t gt_cta = __reduce_add_sync(0xffffffffu, gt_all), eq_cta = __reduce_add_sync(0xffffffffu, eq_all);
        if (lane < CS) {
          peer_store(peer_address(&sh.cta_gt[si][rank], (uint32_t)lane), gt_cta);
          peer_store(peer_address(&sh.cta_eq[si][rank], (uint32_t)lane), eq_cta);
        }
      }
      cluster_barrier();
      gt_before += __reduce_add_sync(0xffffffffu, lane < rank ? sh.cta_gt[si][lane] : 0u);
      eq_before += __reduce_add_sync(0xffffffffu, lane < rank ? sh.cta_eq[si][lane] : 0u);
    }
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool mine = (in >> j & 1u) != 0u, gt = mine && key[j] > thr, eq = mine && key[j] == thr;
      const uint32_t m_gt = __ballot_sync(0xffffffffu, gt), m_eq = __ballot_sync(0xffffffffu, eq);
      const uint32_t eq_rank = eq_before + __popc(m_eq & below);              // ties go to the lowest positions
      if (gt || (eq && eq_rank < need_eq)) emit((int)(run_out + gt_before + __popc(m_gt & below) + min(eq_rank, need_eq)), c0 + 32 * j);
      gt_before += __popc(m_gt);
      eq_before += __popc(m_eq);
    }
    run_out += (uint32_t)n;
  }
}

// The keys of a thread's items: candidates c0 + 32 j below c_end.
template <int KPT>
__device__ __forceinline__ void load_keys(uint32_t (&key)[KPT], const float* scores, const HeadPlace& h, int kpt, int c0, int c_end) {
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int c = c0 + 32 * j;
    key[j] = 0u;
    if (j < kpt && c < c_end) key[j] = score_key(__ldcg(scores + (c < h.o ? c : c + h.b)));
  }
}

struct GatherHead {                       // the rows of one (sequence, KV head)
  const char *k, *v;
  char *k_c, *v_c;
};
__device__ __forceinline__ GatherHead gather_head(const CompactParams& p, int bi, int g) {
  return {reinterpret_cast<const char*>(p.k) + bi * p.kv_stride_bytes[0] + g * p.kv_stride_bytes[1],
          reinterpret_cast<const char*>(p.v) + bi * p.kv_stride_bytes[0] + g * p.kv_stride_bytes[1],
          reinterpret_cast<char*>(p.k_c) + bi * p.c_stride_bytes[0] + g * p.c_stride_bytes[1],
          reinterpret_cast<char*>(p.v_c) + bi * p.c_stride_bytes[0] + g * p.c_stride_bytes[1]};
}

// Stages of 16 bytes of K and of V per thread that fit `bytes`.
__host__ __device__ constexpr int gather_stages(int nt, int bytes) { return bytes / (32 * nt); }
// Copies the rows of the kept entries [i_lo, i_hi), whose positions are kept_s[0 ..), into the compacted cache. The rows pass through
// shared memory, where every thread keeps its own 16-byte pieces, one of K and one of V per stage and STAGES on their way at a time,
// without holding them in registers and without a barrier: for CTAs of few threads and registers beside another kernel's. (Alone
// on its SM a CTA of 1024 threads with eight pieces each in registers is ahead: 32 heads x 1280 keys, attention and this one after
// the other 20.1 us, 21.9 with 384 threads and 96 KB of stages.)
template <int NT, int STAGES>
__device__ __forceinline__ void gather_rows(const CompactParams& cp, const GatherHead& gh, unsigned char* stages_s, const int32_t* kept_s, int i_lo, int i_hi) {
  const int tid = threadIdx.x, lg = 31 - __clz(cp.row_bytes / 16);        // log2 of the threads per row
  const int rows_per_pass = NT >> lg, c16 = tid & ((1 << lg) - 1), passes = (i_hi - i_lo + rows_per_pass - 1) / rows_per_pass;
  uint4* mine = reinterpret_cast<uint4*>(stages_s) + tid;                 // [stage][K, V][thread]
  auto fetch = [&](int pass, int stage) {
    const int i = i_lo + pass * rows_per_pass + (tid >> lg);
    if (i < i_hi) {
      const int64_t at = (int64_t)kept_s[i - i_lo] * cp.kv_stride_bytes[2] + c16 * 16;
      dev::cp_async16(dev::smem_u32(mine + stage * 2 * NT), gh.k + at, 16);
      dev::cp_async16(dev::smem_u32(mine + (stage * 2 + 1) * NT), gh.v + at, 16);
    }
    dev::cp_async_commit();
  };
#pragma unroll
  for (int st = 0; st < STAGES; ++st) fetch(st, st);
#pragma unroll 1
  for (int p0 = 0; p0 < passes; p0 += STAGES) {
#pragma unroll
    for (int st = 0; st < STAGES; ++st) {
      dev::cp_async_wait<STAGES - 1>();
      const int i = i_lo + (p0 + st) * rows_per_pass + (tid >> lg);
      if (i < i_hi) {
        reinterpret_cast<uint4*>(gh.k_c + (int64_t)i * cp.c_stride_bytes[2])[c16] = mine[st * 2 * NT];
        reinterpret_cast<uint4*>(gh.v_c + (int64_t)i * cp.c_stride_bytes[2])[c16] = mine[(st * 2 + 1) * NT];
      }
      fetch(p0 + st + STAGES, st);
    }
  }
}

// The head's raw saliency in shared memory by candidate, with room for half a window in front, behind and, per region, between the
// regions: with the neutral value there (-inf, or 0 for averages) a window needs no look at the ends of its axis.
struct RawAxis {
  int w, gap, o, kind, window;    // half window; its width again between the regions, or 0; candidates in front of the block
  __device__ __forceinline__ RawAxis(const SelectParams& p, const HeadPlace& h)
      : w((p.window - 1) / 2), gap(p.mode != SDLLM_SELECT_JOINT_FLOOR ? w : 0), o(h.o), kind(p.pool_kind), window(p.window) {}
  __device__ __forceinline__ int at(int c) const { return w + c + (c >= o ? gap : 0); }
  __device__ __forceinline__ void clear_ends(float* raw, int C, int t, int nt) const {
    const float none = kind == SDLLM_POOL_MAX ? -INFINITY : 0.f;
    for (int i = t; i < w; i += nt) {
      raw[i] = none;
      raw[w + C + gap + i] = none;
      if (gap > 0) raw[w + o + i] = none;
    }
  }
  // Algorithm 1, MaxPool1D(A, kernel_size = s, padding = s/2) over the candidate axis. W > 0: half windows of at most W, all reads of
  // which go out together.
  template <int W>
  __device__ __forceinline__ float pool(const float* raw, int c) const {
    const float* x = raw + at(c);
    float mx = -INFINITY, sum = 0.f;
    if constexpr (W > 0) {
#pragma unroll
      for (int k = -W; k <= W; ++k) {
        const float v = k >= -w && k <= w ? x[k] : (kind == SDLLM_POOL_MAX ? -INFINITY : 0.f);
        mx = fmaxf(mx, v);
        sum += v;
      }
    } else {
      for (int k = -w; k <= w; ++k) {
        mx = fmaxf(mx, x[k]);
        sum += x[k];
      }
    }
    return kind == SDLLM_POOL_MAX ? mx : sum / (float)window;
  }
};
__host__ __device__ constexpr int raw_axis_floats(int Lmax, int b, int window) { return Lmax - b + 3 * ((window - 1) / 2); }

template <int W, int KPT>
__device__ __forceinline__ void pool_keys(uint32_t (&key)[KPT], const RawAxis& axis, const float* raw, int C, int kpt, int c0) {
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int c = c0 + 32 * j;
    key[j] = 0u;
    if (j < kpt && c < C) key[j] = score_key(axis.pool<W>(raw, c));
  }
}
template <int KPT>
__device__ __forceinline__ void pool_keys(uint32_t (&key)[KPT], const RawAxis& axis, const float* raw, int C, int kpt, int c0) {
  if (axis.w <= 1) pool_keys<1>(key, axis, raw, C, kpt, c0);
  else if (axis.w <= 4) pool_keys<4>(key, axis, raw, C, kpt, c0);
  else pool_keys<0>(key, axis, raw, C, kpt, c0);
}

// The empty entries [z_lo, z_hi) of a head's list and their zero rows, by thread t of nt.
__device__ __forceinline__ void write_empty_entries(const CompactParams& cp, const GatherHead& gh, int32_t* out, int z_lo, int z_hi, int t, int nt) {
  for (int i = z_lo + t; i < z_hi; i += nt) out[i] = -1;
  const int lg = 31 - __clz(cp.row_bytes / 16);        // log2 of the threads per row
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  for (int i = z_lo + (t >> lg); i < z_hi; i += nt >> lg) {
    reinterpret_cast<uint4*>(gh.k_c + (int64_t)i * cp.c_stride_bytes[2])[t & ((1 << lg) - 1)] = zero;
    reinterpret_cast<uint4*>(gh.v_c + (int64_t)i * cp.c_stride_bytes[2])[t & ((1 << lg) - 1)] = zero;
  }
}

// CTA r's share of the head's pooled scores, pooled from the raw ones in shared memory, by thread t of nt.
__device__ __forceinline__ void write_pooled(const SelectParams& p, const float* raw, const HeadPlace& h, int64_t head, int r, int R, int t, int nt) {
  const RawAxis axis(p, h);
  const int p_hi = (int)((int64_t)(r + 1) * p.Lmax / R);
  for (int pos = (int)((int64_t)r * p.Lmax / R) + t; pos < p_hi; pos += nt) {
    const bool candidate = pos < h.o || (pos >= h.o + h.b && pos < h.C + h.b);
    p.pooled_out[head * p.Lmax + pos] = candidate ? axis.pool<0>(raw, pos < h.o ? pos : pos - h.b) : -INFINITY;
  }
}

// CTA `part` of f.ctas folds its share of the rows of one (sequence, KV head).
template <int NT>
__device__ __forceinline__ void fold_head(const FoldParams& f, int bg, int bi, int g, int part) {
  const int c4n = f.D / 4, rows = f.row_tiles > 0 ? f.row_tiles * 128 : f.M;
  for (int item = part * NT + (int)threadIdx.x; item < rows * c4n; item += f.ctas * NT) {
    // lanes along the axis that is contiguous in the partial rows
    const int m = f.row_tiles > 0 ? item / (128 * c4n) * 128 + item % 128 : item / c4n;
    const int c4 = f.row_tiles > 0 ? item / 128 % c4n : item % c4n;
    if (m >= f.M) continue;
    dev::FoldedColumn x;
    if (f.row_tiles > 0) {
      const int64_t first = ((int64_t)bg * f.row_tiles + (m >> 7)) * f.splits;
      const float4* po = reinterpret_cast<const float4*>(f.part_o) + (first * c4n + c4) * 128 + (m & 127);
      const float2* pm = reinterpret_cast<const float2*>(f.part_ml) + first * 128 + (m & 127);
      x = dev::fold_splits<6>(f.splits, [&](int s) { return __ldcg(pm + s * 128); }, [&](int s) { return __ldcg(po + (int64_t)s * c4n * 128); }, fast_exp2);
    } else {
      const float4* po = reinterpret_cast<const float4*>(f.part_o) + ((int64_t)bg * f.splits * f.M + m) * c4n + c4;
      const float2* pm = reinterpret_cast<const float2*>(f.part_ml) + (int64_t)bg * f.splits * f.M + m;
      x = dev::fold_splits<6>(f.splits, [&](int s) { return __ldcg(pm + (int64_t)s * f.M); }, [&](int s) { return __ldcg(po + (int64_t)s * f.M * c4n); },
                              [](float e) { return exp2f(e); });
    }
    const float inv = x.l != 0.f ? 1.f / x.l : 0.f;
    const int hg = m / f.b, i = m - hg * f.b, hq = g * f.G + hg;
    const int64_t off = (int64_t)bi * f.o_stride[0] + (int64_t)hq * f.o_stride[1] + (int64_t)i * f.o_stride[2] + c4 * 4;
    if (f.dtype == SDLLM_BF16)
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(f.out) + off) = make_uint2(dev::pack_bf16(x.o.x * inv, x.o.y * inv), dev::pack_bf16(x.o.z * inv, x.o.w * inv));
    else
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(f.out) + off) = make_float4(x.o.x * inv, x.o.y * inv, x.o.z * inv, x.o.w * inv);
    if (c4 == 0 && f.lse) f.lse[((int64_t)bi * f.Hq + hq) * f.b + i] = (x.m + log2f(x.l)) * kLn2;
  }
}

struct LaunchConfig {                     // a launch with its attributes, which the configuration points to
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  LaunchConfig(dim3 grid, int threads, size_t smem, cudaStream_t st) {
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
  }
  void cluster(int n) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = n; attr[cfg.numAttrs].val.clusterDim.y = 1; attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  void after_start_of_previous() {        // may start while the kernel in front finishes
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    ++cfg.numAttrs;
  }
};
