// Device-side building blocks shared by the tcgen05 attention kernels: PTX wrappers (mbarrier, TMA, tcgen05, TMEM,
// clusters), the shared-memory and instruction descriptors of tcgen05.mma, and the bounded mbarrier waits.
// Meant to be included inside `namespace sdllm { namespace { ... } }` of a .cu file.
#pragma once

constexpr long long kDrainCycles = 400000000LL;   // ~0.2 s: limit of the waits that let in-flight work land on the way out

// ---------------------------------------------------------------------------------------------------------
// PTX wrappers
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// ... without the suspension that try_wait may take while the phase is open
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int x, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];\n"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];\n" ::"l"(tm) : "memory");
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// One lane of a converged warp: the code around it stays warp-uniform, so descriptors are computed in uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (base lane + i)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;\n" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// The larger and the smaller of two, NaN when either is.
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;\n" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;\n" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;\n" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// Two fp32 operations per instruction (same rounding as the scalar forms).
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;\n" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add_f2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// 2^x for two values on the FMA pipe, beside the exponential unit (16 results per clock and SM, the bottleneck of a softmax
// that feeds tcgen05): x = n + f with n the nearest integer (round by adding 1.5 * 2^23), 2^f by the degree-5 polynomial of
// least relative error on [-1/2, 1/2] with 1 as its constant term, its coefficients rounded to fp32 one after the other and the rest
// fitted again (9.4e-8, 1.5e-7 evaluated in fp32, as much as ex2.approx shows; with a free constant term, which rounds to 1 + 2^-23,
// it was 2.1e-7), n added to the exponent. Values below 2^-126 come out as about 2^-126 instead of 0. NaN stays NaN up to the integer addition, which
// makes the largest float of it: a row's sum of exponentials that reaches kNanSum has met one (ordinary sums stay below 2^8 a key).
constexpr float kNanSum = 1e38f;
__device__ __forceinline__ void poly_exp2(float x0, float x1, float& e0, float& e1) {
  const uint64_t x = pack_f2(max_nan(x0, -126.f), max_nan(x1, -126.f));
  const uint64_t magic = pack_f2(12582912.f, 12582912.f), minus_one = pack_f2(-1.f, -1.f);
  const uint64_t t = add_f2(x, magic);
  const uint64_t f = add_f2(x, fma_f2(t, minus_one, magic));
  uint64_t y = fma_f2(pack_f2(1.3256072998046875e-3f, 1.3256072998046875e-3f), f, pack_f2(9.671226143836975e-3f, 9.671226143836975e-3f));
  y = fma_f2(y, f, pack_f2(5.5507682263851166e-2f, 5.5507682263851166e-2f));
  y = fma_f2(y, f, pack_f2(2.402224838733673e-1f, 2.402224838733673e-1f));
  y = fma_f2(y, f, pack_f2(6.931469440460205e-1f, 6.931469440460205e-1f));
  y = fma_f2(y, f, pack_f2(1.f, 1.f));
  float y0, y1, t0, t1;
  unpack_f2(y, y0, y1);
  unpack_f2(t, t0, t1);
  e0 = __uint_as_float(__float_as_uint(y0) + (__float_as_uint(t0) << 23));
  e1 = __uint_as_float(__float_as_uint(y1) + (__float_as_uint(t1) << 23));
}
__device__ __forceinline__ void regs_dec_72() { asm volatile("setmaxnreg.dec.sync.aligned.u32 72;\n"); }
__device__ __forceinline__ void regs_dec_80() { asm volatile("setmaxnreg.dec.sync.aligned.u32 80;\n"); }
__device__ __forceinline__ void regs_inc_208() { asm volatile("setmaxnreg.inc.sync.aligned.u32 208;\n"); }

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}

// Shared-memory matrix descriptor of tcgen05.mma: 128-byte swizzle, start address / leading / stride offsets in
// 16-byte units, descriptor version 1 in bits 46-47, swizzle mode 2 (128 B) in bits 61-63.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, M = 128, N = n, A K-major, B K- or MN-major.
__device__ __forceinline__ uint32_t instr_desc(int n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

// The sequence of rank `rank` when a batch of at most 64 is ordered from the longest to the shortest (equal lengths in batch
// order). A whole warp calls this; every lane gets the answer.
__device__ __forceinline__ int sequence_of_rank(const int32_t* lengths, int B, int rank) {
  const int lane = threadIdx.x & 31;
  const int l0 = lane < B ? lengths[lane] : -1, l1 = lane + 32 < B ? lengths[lane + 32] : -1;
  int r0 = 0, r1 = 0;                                  // how many sequences come before mine
  for (int i = 0; i < B; ++i) {
    const int li = __shfl_sync(0xffffffffu, i < 32 ? l0 : l1, i & 31);
    r0 += (li > l0 || (li == l0 && i < lane)) ? 1 : 0;
    r1 += (li > l1 || (li == l1 && i < lane + 32)) ? 1 : 0;
  }
  const unsigned hit0 = __ballot_sync(0xffffffffu, lane < B && r0 == rank), hit1 = __ballot_sync(0xffffffffu, lane + 32 < B && r1 == rank);
  return hit0 ? __ffs(hit0) - 1 : (hit1 ? __ffs(hit1) + 31 : rank);
}

// Which tile (source, first row, valid rows, MMA width) a CTA-local ordinal refers to.
struct Tile {
  int src1;      // 1: source 1, 0: source 2
  int row0;      // first row inside its source
  int nv;        // valid rows (0: skip the tile)
  int n_mma;     // nv rounded up to 16
};
__device__ __forceinline__ Tile tile_of(int t, int tiles1, int KT, int KT2, int n1, int n2) {
  Tile x;
  if (t < tiles1) { x.src1 = 1; x.row0 = t * KT; x.nv = min(max(n1 - x.row0, 0), KT); }
  else { x.src1 = 0; x.row0 = (t - tiles1) * KT2; x.nv = min(max(n2 - x.row0, 0), KT2); }
  x.n_mma = (x.nv + 15) & ~15;
  return x;
}

// Bounded wait on an mbarrier phase (`limit` clock cycles). Returns false when the CTA is aborting (this wait or another
// one expired). The first look is test_wait: try_wait there as well made a reuse call 1.3 % slower, a ragged batch's 4 %.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status, int code,
                                         long long limit) {
  if (mbar_test_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (limit > 0) {                                    // (with a limit of zero nothing is waited for: try_wait may suspend for longer than a short wait takes)
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) break;
  }
  *abort_flag = 1;
  atomicExch(status, code);
  return false;
}
// The same for a whole warp: every lane takes the same decision, so warp-synchronous instructions stay converged.
__device__ __forceinline__ bool wait_bar_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status, int code,
                                              long long limit) {
  return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag, status, code, limit)) != 0;
}
// Bounded wait that ignores the abort flag (used while draining in-flight work on the way out).
__device__ __forceinline__ void drain_bar(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kDrainCycles) return;
  }
}
// The way out of a CTA in which a wait gave up: what was issued must have landed before the CTA's shared and tensor memory are
// handed on. The abort flag is looked at behind a barrier that all waits lie in front of (a wait of any warp may be the one that
// gives up, also when the producer and the MMA warp are through). The key-row kernel has it where the accumulators have been read,
// while the MMA warp is idle; at its very end the look cost 0.06 of 7.4 us per reuse call.
// Loads of tiles into a ring: the last use of every slot, `full` its first barrier, `issued` the tiles whose load is under way.
__device__ __forceinline__ void drain_loads(uint32_t full, int issued, int slots) {
  for (int j = max(issued - slots, 0); j < issued; ++j) drain_bar(full + 8u * (uint32_t)(j % slots), (uint32_t)(j / slots) & 1u);
}
// MMAs: called by the whole warp that issued them (the election always picks the same lane).
__device__ __forceinline__ void drain_mmas(uint32_t bar) {
  if (elect_one()) {
    tc_commit(bar);
    drain_bar(bar, 0);
  }
  __syncwarp();
}
