// Thin inline-PTX wrappers for the sm_100a features the attention kernels use:
// mbarrier with bounded waits, TMA tiled copies, tcgen05 tensor-core MMA with
// TMEM accumulators, and the shared-memory / instruction descriptors they take.
//
// Every wait here is bounded: after the wait limit (about a second by default) without
// completion the waiter raises a CTA-wide abort flag and stores a code that names the
// wait in the caller's status word; all later waits return at once, no role starts new
// work (the loops over work items and, in the producers, over tiles test the flag), copies
// and tensor-core work in flight are drained, and the kernel returns.  A bug in a barrier
// phase therefore cannot leave the GPU spinning.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace pc {

constexpr unsigned SPIN_BACKOFF_NS = 20;                 // pause between two polls of a barrier
// Producers, and the epilogue where it waits for a block's statistics, pause much longer: their waits last thousands of
// cycles, a wake-up a few hundred cycles late costs them nothing, and every poll they do not make leaves an issue slot to the
// softmax warp that shares their scheduler (measured when the issuing thread paused as long: 1.2 % on the 128K shape; 640 ns is
// too long, and for the softmax warps themselves 0, 20 or 80 ns make no difference).  The issuers: Cfg::ISSUER_NS in pc_flash.cuh.
constexpr unsigned SERVICE_BACKOFF_NS = 320;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ------------------------------------------------------------------ mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// What a bounded wait looks at after every 64 polls: whether it is over without completion.  Out of line: there are some fifty
// waits in a kernel, all its warps share the instruction caches, and these lines at every one of them cost (us in loops of 15 ms, in
// line / out of line) head size 64, 8 chunks of 4096, 32/8 heads 877 / 857, 22 of 958 259 / 249; head size 128, 3 of 2372, 28/4 heads
// 188 / 179, 5 of 298 42.5 / 41.1; window of 16 over 64 caches of 16000, head size 64 496 / 478; a decoding step over one cache of
// 16401 15.7 / 15.6; at the power cap (8 of 8192, 32/8 heads of 128 4018 / 4034) nothing.  What is alive across the call costs the roles
// registers: spills stored, bytes, prefill 20 / 48 at head size 64, 28 / 48 at 128 on pairs, query windows 0 / 16 to 24 (in those times).
static __device__ __noinline__ bool mbar_wait_over(long long t0, volatile int* abort_flag, int* status_word, int where) {
  if (*abort_flag) return true;
  if (clock64() - t0 <= (static_cast<long long>(abort_flag[1]) << 10)) return false;
  *abort_flag = 1;
  if (status_word) atomicCAS(status_word, 0, where);
  return true;
}

// Bounded wait.  `abort_flag` points at two adjacent ints in shared memory: the CTA's abort
// flag and the wait limit in units of 1024 cycles.  Once the flag is non-zero every wait
// returns immediately (the result data is then garbage and the status word says so).
// Returns false if the wait gave up.
// NS: pause between two polls.
template <unsigned NS>
__device__ __forceinline__ bool mbar_wait_ns(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                             int* status_word, int where) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (NS > 0) __nanosleep(NS);                             // a hot spin takes issue slots from the warps that share the scheduler
    if ((++spins & 63u) == 0u && mbar_wait_over(t0, abort_flag, status_word, where)) return false;
  }
  return true;
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          int* status_word, int where) {
  return mbar_wait_ns<SPIN_BACKOFF_NS>(bar, parity, abort_flag, status_word, where);
}

// Wait that ignores the abort flag (used only to drain copies and tensor-core work in flight before
// exit); gives up after an eighth of the wait limit.
__device__ __forceinline__ void mbar_wait_drain(uint64_t* bar, uint32_t parity, const volatile int* abort_flag) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > (static_cast<long long>(abort_flag[1]) << 7)) return;
  }
}
// After an abort: a fixed pause (a tenth of a millisecond) that outlasts any copy this CTA may still have in
// flight towards its shared memory whose completion it cannot observe on a barrier of its own.
__device__ __forceinline__ void abort_grace_pause(const volatile int* abort_flag) {
  if (*abort_flag == 0) return;
  const long long t0 = clock64();
  while (clock64() - t0 < 200000LL) __nanosleep(1000);
}

// ------------------------------------------------------------------ fences
__device__ __forceinline__ void fence_proxy_async_smem() {   // generic-proxy smem writes -> async proxy (TMA / MMA)
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void named_barrier_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// ------------------------------------------------------------------ TMA (tiled, 4-D)
// Coordinates are innermost first.  The innermost coordinate times the element
// size must be a multiple of 16 bytes (callers only pass multiples of 64 elements).
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const void* tmap, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d_addr(void* smem_dst, const void* tmap, uint32_t bar_addr, int c0, int c1, int c2,
                                                 int c3) {        // barrier given by its shared-memory address
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(bar_addr), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_store_4d(const void* tmap, const void* smem_src, int c0, int c1, int c2,
                                             int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(tmap),
               "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() {   // smem source may be reused
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void tma_store_wait_all() {    // writes complete
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
// one 32-byte store (a whole sector: rows that threads write each on their own); p aligned to 32 bytes
__device__ __forceinline__ void st_global_f32x8(void* p, const float* x) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               :: "l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7]) : "memory");
}
__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}

// ------------------------------------------------------------------ TMEM
// One warp allocates `ncols` (power of two >= 32) columns; the base address is
// written to shared memory.  The same warp frees them.
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 32 lanes x 32 columns of 32-bit: thread i of the warp receives lane (base_lane + i),
// register j holds column (base_col + j).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------------ descriptors
// Shared-memory matrix descriptor, 128-byte swizzle.  The tile is stored as rows
// of 128 bytes (64 bf16); 8 consecutive rows form one 1024-byte swizzle atom.
//   K-major operand  (rows = M or N index, the 64 elements of a row run along K):
//       SBO = 1024 (next 8 rows); LBO unused.
//   MN-major operand (rows = K index, the 64 elements of a row run along M or N):
//       SBO = 1024 (next 8 K rows); LBO = byte distance to the next block of 64 M/N elements.
__device__ __forceinline__ uint64_t make_smem_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes,
                                                         uint32_t sbo_bytes) {
  uint64_t desc = 0;
  desc |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
  desc |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
  desc |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
  desc |= static_cast<uint64_t>(1) << 46;    // descriptor version for sm_100
  desc |= static_cast<uint64_t>(2) << 61;    // SWIZZLE_128B
  return desc;
}

// Instruction descriptor for kind::f16 with bf16 operands and fp32 accumulation.
__host__ __device__ constexpr uint32_t make_idesc_bf16_f32(int M, int N, bool a_mn_major, bool b_mn_major) {
  return (1u << 4)                                   // D format: f32
         | (1u << 7)                                 // A format: bf16
         | (1u << 10)                                // B format: bf16
         | (static_cast<uint32_t>(a_mn_major) << 15)
         | (static_cast<uint32_t>(b_mn_major) << 16)
         | (static_cast<uint32_t>(N >> 3) << 17)
         | (static_cast<uint32_t>(M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]; issued by ONE thread.
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(static_cast<uint32_t>(accumulate))
      : "memory");
}
// Arrive on an mbarrier once every tcgen05 operation issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// ------------------------------------------------------------------ small helpers
// Byte offset of the 16-byte chunk `chunk` (0..7) of row `row` inside a 128-byte-swizzled
// tile whose rows are 128 bytes: the chunk index is XOR-ed with the row index modulo 8.
__device__ __forceinline__ uint32_t sw128_offset(uint32_t row, uint32_t chunk) {
  return row * 128u + ((chunk ^ (row & 7u)) << 4);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ------------------------------------------------------------------ packed fp32 pairs and 3-input max (sm_100)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {   // a * b + c on both halves
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Round an fp64 value to bf16, ties to even, in one rounding (no fp32 detour).
__device__ __forceinline__ uint16_t f64_to_bf16_rne(double x) {
  // fp64 -> fp32 with round-to-odd keeps enough information for a second, exact RNE step
  float f = __double2float_rz(x);
  if (static_cast<double>(f) != x) f = __uint_as_float(__float_as_uint(f) | 1u);   // sticky bit
  uint32_t u = __float_as_uint(f);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return static_cast<uint16_t>(u >> 16);
}

// ------------------------------------------------------------------ CTA pairs (cluster of 2, cta_group::2)
// One tcgen05.mma with cta_group::2 computes a 256-row product across two SMs: each CTA
// supplies its own 128 rows of A (shared memory or TMEM) and HALF of the N extent of B at the
// same shared-memory offset; the accumulator rows of a CTA land in its own TMEM.  The
// instruction is issued by one thread of the leader CTA (cluster rank 0).
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {       // every thread of both CTAs
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(const void* local_smem, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local_smem)), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {   // barrier may live in the peer CTA
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Same signal without cluster-scope release: for barriers that guard TMEM or async-proxy data, whose
// ordering comes from tcgen05.fence / fence.proxy.async, not from generic memory ordering.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// wait with cluster-scope acquire (data written by the peer CTA before its release-arrive is visible)
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// TMA load into this CTA's shared memory whose completion bytes are counted on a barrier
// that may live in the peer CTA of the pair (no multicast: every CTA fetches its own half).
__device__ __forceinline__ void tma_load_4d_pair(void* smem_dst, const void* tmap, uint32_t bar_cluster_addr, int c0,
                                                 int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(bar_cluster_addr), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_result, uint32_t ncols) {   // one warp in EACH CTA
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Arrive on the barrier at this shared-memory offset in BOTH CTAs once every tcgen05
// operation issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(3))
               : "memory");
}

// One thread of a converged warp (elect.sync).  Unlike `lane == 0` the compiler knows that the branch is taken by a
// single thread, and keeps the operands of tcgen05 instructions in uniform registers: issuing the eight k-steps of a
// 128 x 128 x 128 product takes 121 to 200 cycles in such a branch and 410 to 470 under `lane == 0`.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
template <int N> __device__ __forceinline__ void setmaxnreg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void setmaxnreg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// ------------------------------------------------------------------ whole products as one asm block
// The k-steps of a product are one asm statement whose descriptors differ by immediates in the low word (121 cycles to
// issue the eight steps, against 200 for eight statements under elect_one), so that the issuing thread stays ahead of
// the pipe, which needs 512 cycles for them.  Operand tiles: rows of 64 elements, 128-byte swizzle; a k-step is 16
// elements = 32 bytes, the next 64 elements of a row are an atom of 8 KB (64 rows) or 16 KB (128 rows) further.
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);        // SBO 1024, sm_100 descriptor, 128-byte swizzle
__device__ __forceinline__ uint32_t desc_lo(uint32_t smem, uint32_t lbo) { return ((smem & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16); }
#define PC_MMA_SS0(G) "setp.ne.b32 p, 0, 0;\n\tmov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\ttcgen05.mma.cta_group::" #G ".kind::f16 [%0], a, b, %4, p;\n\tsetp.eq.b32 p, 0, 0;\n\t"
#define PC_MMA_SS(G, oa, ob) "add.s32 x, %1, " #oa ";\n\tadd.s32 y, %2, " #ob ";\n\tmov.b64 a, {x, %3};\n\tmov.b64 b, {y, %3};\n\ttcgen05.mma.cta_group::" #G ".kind::f16 [%0], a, b, %4, p;\n\t"
#define PC_MMA_TS(G, t, o) "add.s32 x, %1, " #t ";\n\tadd.s32 y, %2, " #o ";\n\tmov.b64 b, {y, %3};\n\ttcgen05.mma.cta_group::" #G ".kind::f16 [%0], [x], b, %4, p;\n\t"
#define PC_SS_REGS "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t.reg .b32 x, y;\n\t"
// S = A B^T over 64 elements (one atom), single CTA
__device__ __forceinline__ void mma_ss_k64(uint32_t d_tmem, uint32_t a_smem, uint32_t b_smem, uint32_t idesc) {
  asm volatile(PC_SS_REGS PC_MMA_SS0(1) PC_MMA_SS(1, 2, 2) PC_MMA_SS(1, 4, 4) PC_MMA_SS(1, 6, 6) "}\n"
               ::"r"(d_tmem), "r"(desc_lo(a_smem, 16)), "r"(desc_lo(b_smem, 16)), "r"(DESC_HI), "r"(idesc) : "memory");
}
// the same over 128 elements, operands of 128 rows
__device__ __forceinline__ void mma_ss_k128(uint32_t d_tmem, uint32_t a_smem, uint32_t b_smem, uint32_t idesc) {
  asm volatile(PC_SS_REGS PC_MMA_SS0(1) PC_MMA_SS(1, 2, 2) PC_MMA_SS(1, 4, 4) PC_MMA_SS(1, 6, 6)
               PC_MMA_SS(1, 1024, 1024) PC_MMA_SS(1, 1026, 1026) PC_MMA_SS(1, 1028, 1028) PC_MMA_SS(1, 1030, 1030) "}\n"
               ::"r"(d_tmem), "r"(desc_lo(a_smem, 16)), "r"(desc_lo(b_smem, 16)), "r"(DESC_HI), "r"(idesc) : "memory");
}
// S = A B^T over 128 elements on a CTA pair; A 128 rows per CTA, B 64 rows (B64) or up to 128 rows per CTA
template <bool B64>
__device__ __forceinline__ void mma_ss_pair_k128(uint32_t d_tmem, uint32_t a_smem, uint32_t b_smem, uint32_t idesc) {
  if constexpr (B64)
    asm volatile(PC_SS_REGS PC_MMA_SS0(2) PC_MMA_SS(2, 2, 2) PC_MMA_SS(2, 4, 4) PC_MMA_SS(2, 6, 6)
                 PC_MMA_SS(2, 1024, 512) PC_MMA_SS(2, 1026, 514) PC_MMA_SS(2, 1028, 516) PC_MMA_SS(2, 1030, 518) "}\n"
                 ::"r"(d_tmem), "r"(desc_lo(a_smem, 16)), "r"(desc_lo(b_smem, 16)), "r"(DESC_HI), "r"(idesc) : "memory");
  else
    asm volatile(PC_SS_REGS PC_MMA_SS0(2) PC_MMA_SS(2, 2, 2) PC_MMA_SS(2, 4, 4) PC_MMA_SS(2, 6, 6)
                 PC_MMA_SS(2, 1024, 1024) PC_MMA_SS(2, 1026, 1026) PC_MMA_SS(2, 1028, 1028) PC_MMA_SS(2, 1030, 1030) "}\n"
                 ::"r"(d_tmem), "r"(desc_lo(a_smem, 16)), "r"(desc_lo(b_smem, 16)), "r"(DESC_HI), "r"(idesc) : "memory");
}
// four k-steps (64 keys) of O (+)= P V, P in TMEM; p_tmem and v_smem point at the first of them
template <bool PAIR>
__device__ __forceinline__ void mma_ts_k64(uint32_t o_tmem, uint32_t p_tmem, uint32_t v_smem, uint32_t idesc, bool accumulate) {
  if constexpr (PAIR)
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t.reg .b32 x, y;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 b, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], b, %4, p;\n\tsetp.eq.b32 p, 0, 0;\n\t"
                 PC_MMA_TS(2, 8, 128) PC_MMA_TS(2, 16, 256) PC_MMA_TS(2, 24, 384) "}\n"
                 ::"r"(o_tmem), "r"(p_tmem), "r"(desc_lo(v_smem, 16384)), "r"(DESC_HI), "r"(idesc), "r"(static_cast<uint32_t>(accumulate)) : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t.reg .b32 x, y;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 b, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n\tsetp.eq.b32 p, 0, 0;\n\t"
                 PC_MMA_TS(1, 8, 128) PC_MMA_TS(1, 16, 256) PC_MMA_TS(1, 24, 384) "}\n"
                 ::"r"(o_tmem), "r"(p_tmem), "r"(desc_lo(v_smem, 16384)), "r"(DESC_HI), "r"(idesc), "r"(static_cast<uint32_t>(accumulate)) : "memory");
}

// 32-bit store into the shared memory of a CTA of the cluster whose completion is counted (4 bytes) on an mbarrier there
__device__ __forceinline__ void st_async_u32(uint32_t cluster_addr, uint32_t v, uint32_t bar_cluster_addr) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(cluster_addr), "r"(v),
               "r"(bar_cluster_addr)
               : "memory");
}

}  // namespace pc
