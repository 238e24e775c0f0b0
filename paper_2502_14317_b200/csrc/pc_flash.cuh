// What the flash-attention kernels on two query blocks per CTA share (chunk-local attention, pc_prefill2.cu; parallel
// attention, pc_parallel.cu): roles, shared-memory layout, barriers, work descriptors, the K/V ring, MMA issue.
//
// A CTA owns two 128-row query blocks A and B, one softmax warpgroup each; while the softmax of one runs the tensor
// cores work for the other.  Warps (16): 0-3 softmax of block A, 4-7 softmax of block B (thread = query row = TMEM lane),
// 8-11 epilogue (the softmax warps go straight on to the next block), 12 TMA producer, 13 issuer of S = Q K^T and of the score
// sweeps, 14 issuer of O += P V (of a CTA pair: in the leader only), 15 idle.  Registers are dealt out by role.
// The issuers are two because their waits have nothing to do with each other: S is due when the S before it has been read,
// P V when P arrives.  One thread in a fixed order was busy for two thirds of a step and late for both.  In a loop, us, one
// thread / two (and, in the prefill, the registers below): 8 chunks of 8192, 32/8 heads 3924 / 3865, 8 of 4096, 32/32 heads
// 1346 / 1333, 4 of 1257, 32/32 heads 138.1 / 135.8; query windows: pc_parallel.cu.
// Keys and values have rings of their own, so that each of them is consumed by one issuer (of a pair's value ring the sweeps
// take stages too).
//
// Tensor memory, 512 columns.  Head size 128: one S (128), P of both blocks (64 each), both accumulators (128 each).  The
// blocks take turns on S: the softmax warps take a whole S into registers at once, and the product for the other block runs
// under their exponentials.  A block therefore finds its next S ready when it is through with a tile, and the blocks'
// exponentials are kept half a step apart.  (With an S of its own for each block and P over its first half, the next product
// waited for P V of the tile before, 1000 of 3300 cycles a step.)  Head size 64, whose accumulators take half the columns: an
// S of each block and P beside them, so that no block waits for the other to read (prefill in a loop, one S / two, us: 8 chunks
// of 4096, 32/32 heads 923 / 909, 22 of 958, 32/8 heads 284 / 278; query windows the same).
// Cfg<D, PAIR>: head size, and whether two CTAs of a cluster work as one unit (cta_group::2: blocks of 2 x 128 rows, every
// K/V tile split between the two shared memories).
#pragma once
#include "pc_softmax.cuh"

namespace pc {
namespace flash {

constexpr int TILE = 128;
constexpr int NT2 = 512;                     // threads per CTA
constexpr int WARP_EPI = 8, WARP_PRODUCER = 12, WARP_QK = 13, WARP_PV = 14;
// Registers by role, 128 * (2 * softmax + epilogue + service) = 64 K.  In a loop, us: prefill, 8 chunks of 8192, 32/8 heads
// 184/80/64 4073, 192/80/48 3983, 192/64/64 3993, 8 of 4096, 32/32 heads 1399 / 1366 / 1378; over caches softmax 184 619, 192 631.
// The service roles spill (-Xptxas -v, bytes stored / loaded at head size 128 on pairs: 48 / 60, spread 72 / 92; with 192/64/64, no
// faster, 32 / 32 and 28 / 28).
struct Regs { int softmax, epilogue, service; };
constexpr Regs REGS_PREFILL = {192, 80, 48}, REGS_PARALLEL = {184, 80, 64};
constexpr int NDESC = 4;                     // work descriptors in flight
constexpr int MAX_NQ = 4, MAX_NS = 6;
template <int D_, bool PAIR_>
struct Cfg {
  static constexpr int D = D_;
  static constexpr bool PAIR = PAIR_;
  static constexpr int NCTA = PAIR ? 2 : 1;
  static constexpr int ATOMS = D / 64;
  static constexpr int Q_BYTES = TILE * D * 2;
  static constexpr int STAGE_BYTES = TILE * D * 2 / NCTA;  // K/V rings: a tile, or of a pair 64 keys of K / half the columns of V
  static constexpr int NQ = STAGE_BYTES == 16384 ? 4 : 2;  // query slots
  static constexpr int NS = STAGE_BYTES == 16384 ? 6 : 5;
  // Stages of keys and of values, alternating.  Of five the values get three: they stay until P has been found, keys only
  // until the next product.  Caches read at the memory's rate, us, 3 + 2 / 2 + 3: window of 16 over 64 caches of 16000, 32/8
  // heads 768 / 735, 64 of 2000 121 / 116, window of 64 over 18 of 8000, 32/32 heads 441 / 421; chunks on single CTAs the same
  // (64 x 384, 32/32 heads 423 / 421).
  static constexpr int NK = NS / 2, NV = NS - NK;
  // TMEM: S of block b (head size 128: one for both in turn), its P at TM_P + 64 b, its accumulator at TM_O + D b
  static constexpr bool TWO_S = D == 64;
  static constexpr uint32_t TM_P = TWO_S ? 256 : 128, TM_O = TWO_S ? 384 : 256;
  static constexpr __host__ __device__ uint32_t tm_s(int b) { return TWO_S ? 128u * b : 0u; }
  // The issuers poll without a pause.  us, 20 ns / none, head size 128, in loops: 8 chunks of 8192, 32/8 heads 4027 / 3989, 2 of 873,
  // 32/32 heads 51.0 / 50.8, 5 of 298, 28/4 heads 41.7 / 41.2, windows of 64 over two caches of 16384 51.2 / 50.5, one of 4096 20.6 / 20.5,
  // 64 of 16384 (power cap) nothing; head size 64, windows of 64 over 32 caches of 8192, 14/2 heads 112.4 / 111.0.
  static constexpr unsigned ISSUER_NS = 0;
  static constexpr int CODE = PAIR ? 200 : 100;            // wait codes in the status word
};

enum { W2_DESC = 1, W2_ITEM, W2_QFULL, W2_QFREE, W2_KVFULL, W2_KVFREE, W2_SFULL, W2_PHALF, W2_PFULL, W2_OFULL, W2_OFREE, W2_LM,
       W2_LMFREE, W2_LSE, W2_TFULL, W2_TFREE, W2_SREAD, W2_PV, W2_SWEEP };

enum { KIND_DONE = 0, KIND_FLASH = 1, KIND_SWEEP = 2 };
struct __align__(16) Desc {
  int kind, c, hkv, len;       // chunk, kv-head, tokens of the chunk
  int h[2], t[2];              // FLASH: q-head and query tile of this CTA's block A / B (t < 0 or behind the chunk: no such
                               // tile, the rows are computed on zeros and not stored);  SWEEP: h[0] = pass
  int n[2];                    // FLASH: key tiles walked for block A / B; 0: block absent (in both CTAs of a pair)
};

struct __align__(16) Misc2 {
  // of a pair: q_full, kv_full, p_*, o_free, t_free, s_read in the leader only; completions of MMAs in both CTAs
  uint64_t q_full[MAX_NQ], q_free[MAX_NQ];
  uint64_t kv_full[MAX_NS], kv_free[MAX_NS];
  uint64_t s_full[2], o_full[2], t_full[2];
  uint64_t p_half[2], p_full[2], o_free[2], t_free[2];
  uint64_t s_read[2], pv_done[2];            // S is in registers (one S: [0]) / P V of a tile has run
  uint64_t lm_full[2], lm_free[2];
  uint64_t d_full[NDESC], d_free[NDESC];
  uint64_t item_full, item_free;             // work items from the leader's producer to its peer's
  uint64_t lse_rdy;
  uint64_t sweep_go;                         // the accumulators have been read out: a score sweep may overwrite them
  uint64_t mma_done;
  Desc desc[NDESC];
  int left[2];                               // warps of the epilogue / the softmax that are through (leave_group)
  int item;
  uint32_t tmem_base;
  int abort_flag;                            // the two words after tmem_base stay adjacent: bounded waits read the limit
  int wait_kcycles;                          // through the flag's address
  alignas(16) float lm[2][2][TILE];          // [block][max / sum][row]: final statistics of a block; in the score sweep [0]:
                                             // [buffer][key] partial window scores of the second column half, [1]:
                                             // [column half][column] log-sum-exp of the window rows
};

template <class C>
struct Off {
  static constexpr int Q = 0, RING = C::NQ * C::Q_BYTES, MISC = RING + C::NS * C::STAGE_BYTES, TOTAL = MISC + (int)sizeof(Misc2);
  static_assert(TOTAL <= 232448, "shared memory of a CTA");
};

__device__ __forceinline__ uint32_t full_par(uint32_t n) { return n & 1u; }           // n-th completion of a barrier
__device__ __forceinline__ uint32_t free_par(uint32_t n) { return (n & 1u) ^ 1u; }    // completion n-1 (passes for n = 0)

struct Ctx2 {
  Misc2* mi;
  uint8_t* sQ;
  uint8_t* ring;
  uint32_t tmem;
  volatile int* abort_flag;
  int* status;
};

// waits of the single-thread service roles (long pause between polls) / of the issuers / of the softmax and epilogue warps
#define WAIT2(bar, par, code) mbar_wait_ns<SERVICE_BACKOFF_NS>((bar), (par), cx.abort_flag, cx.status, C::CODE + (code))
#define WAIT2I(bar, par, code) mbar_wait_ns<C::ISSUER_NS>((bar), (par), cx.abort_flag, cx.status, C::CODE + (code))
#define WAIT2S(bar, par, code) mbar_wait((bar), (par), cx.abort_flag, cx.status, C::CODE + (code))

__device__ __forceinline__ void warp_arrive(uint64_t* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}
// cluster address of the same barrier in CTA `rank` of a pair / of this CTA
template <class C>
__device__ __forceinline__ uint32_t in_cta(const void* p, uint32_t rank) {
  if constexpr (C::PAIR) return map_to_cta(p, rank);
  else return smem_u32(p);
}
template <class C>
__device__ __forceinline__ void commit(uint64_t* bar) {           // in both CTAs of a pair
  if constexpr (C::PAIR) mma_commit_pair(bar);
  else mma_commit(bar);
}
template <class C>
__device__ __forceinline__ void load_box(void* dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2, int c3) {
  if constexpr (C::PAIR) tma_load_4d_pair(dst, tm, bar, c0, c1, c2, c3);
  else tma_load_4d_addr(dst, tm, bar, c0, c1, c2, c3);
}
// one arrival of the warp on a barrier of the leader CTA; guards TMEM data, ordered by the tcgen05 fence
__device__ __forceinline__ void warp_arrive_leader(uint32_t leader_addr) {
  tc_fence_before_sync();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive_remote(leader_addr);
}

// waits until a counter in global memory has reached n (bounded as every wait); the writes before its increments are visible then
__device__ __forceinline__ void wait_count(const int* count, int n, volatile int* abort_flag, int* status, int where) {
  const long long t0 = clock64();
  while (!*abort_flag) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
    if (v >= n) break;
    if (clock64() - t0 > (static_cast<long long>(abort_flag[1]) << 10)) {
      if (status) atomicCAS(status, 0, where);
      *abort_flag = 1;
    }
    __nanosleep(100);
  }
  __threadfence();
}

// wait whose completion also makes the peer CTA's earlier writes visible
__device__ __forceinline__ void mbar_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                                  int where) {
  if (mbar_try_wait_cluster(bar, parity)) return;
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (!mbar_try_wait_cluster(bar, parity)) {
    if ((++spins & 63u) == 0u) {
      if (*abort_flag) return;
      if (clock64() - t0 > (static_cast<long long>(abort_flag[1]) << 10)) {
        *abort_flag = 1;
        if (status) atomicCAS(status, 0, where);
        return;
      }
    }
  }
}

template <class C>
__device__ __forceinline__ void init_barriers2(Misc2& mi, int wait_kcycles, bool leader) {
  constexpr int N = C::NCTA;
  for (int i = 0; i < C::NQ; ++i) { mbar_init(&mi.q_full[i], 1); mbar_init(&mi.q_free[i], 1); }
  for (int i = 0; i < C::NS; ++i) { mbar_init(&mi.kv_full[i], 1); mbar_init(&mi.kv_free[i], 1); }
  for (int b = 0; b < 2; ++b) {
    mbar_init(&mi.s_full[b], 1); mbar_init(&mi.o_full[b], 1); mbar_init(&mi.t_full[b], 1);
    mbar_init(&mi.p_half[b], 4 * N); mbar_init(&mi.p_full[b], 4 * N); // 4 softmax warps of the block in each CTA
    mbar_init(&mi.o_free[b], 4 * N); mbar_init(&mi.t_free[b], 8 * N); // epilogue warps / softmax warps of the CTAs
    mbar_init(&mi.s_read[b], 4 * N); mbar_init(&mi.pv_done[b], 1);
    mbar_init(&mi.lm_full[b], 4); mbar_init(&mi.lm_free[b], 4);
  }
  for (int i = 0; i < NDESC; ++i) { mbar_init(&mi.d_full[i], 1); mbar_init(&mi.d_free[i], leader ? 14 : 12); }   // warps, issuers
  mbar_init(&mi.item_full, 1); mbar_init(&mi.item_free, 1);
  mbar_init(&mi.lse_rdy, 4 * N);
  mbar_init(&mi.sweep_go, 1);
  mbar_init(&mi.mma_done, 2);
  mi.left[0] = mi.left[1] = 0;
  mi.abort_flag = 0;
  mi.wait_kcycles = wait_kcycles;
  fence_mbar_init();
}

// consumers of the descriptor ring.  whole_warp: all 32 threads call.
template <class C>
__device__ __forceinline__ Desc next_desc(const Ctx2& cx, uint32_t& n, bool whole_warp) {
  Misc2& mi = *cx.mi;
  const int slot = n % NDESC;
  Desc d;
  if (!WAIT2S(&mi.d_full[slot], full_par(n / NDESC), W2_DESC) || *cx.abort_flag) { d.kind = KIND_DONE; return d; }
  d = mi.desc[slot];
  if (whole_warp) warp_arrive(&mi.d_free[slot]); else mbar_arrive(&mi.d_free[slot]);
  ++n;
  return d;
}

// A warp of a group that meets at hardware barrier `id` leaves its loop.  After a wait has run out the warps of a group see the abort
// flag at different times: one may leave while another goes on to such a barrier, which has no limit.  So a warp that is
// through keeps meeting the others there until all are through.  Every warp takes part in every meeting, so that they
// agree on its number (odd: whether this warp has taken part in an odd number so far): arrivals are counted after an even one and
// looked at after an odd one, and all see the same count.
template <int WARPS>
__device__ __forceinline__ void leave_group(int id, bool odd, int* left) {
  if (odd) named_barrier_sync(id, 32 * WARPS);
  if ((threadIdx.x & 31) == 0) atomicAdd(left, 1);
  __syncwarp();
  while (true) {
    named_barrier_sync(id, 32 * WARPS);
    const bool all = *reinterpret_cast<volatile int*>(left) == WARPS;
    if (all) break;
    named_barrier_sync(id, 32 * WARPS);
  }
}

// ------------------------------------------------------------------ producer
struct Prod { uint32_t k = 0, v = 0, q = 0, d = 0, item = 0; };
template <class C>
__device__ __forceinline__ void publish(const Ctx2& cx, Prod& p, const Desc& d, bool signal = true) {
  Misc2& mi = *cx.mi;
  const int slot = p.d % NDESC;
  WAIT2(&mi.d_free[slot], free_par(p.d / NDESC), W2_DESC);
  mi.desc[slot] = d;
  if (signal) mbar_arrive(&mi.d_full[slot]);
  ++p.d;
}
// The leader's producer draws items from the queue and hands each to its peer's.
template <class C>
__device__ __forceinline__ int next_item(const Ctx2& cx, Prod& p, bool leader, int* counter, int n_items) {
  Misc2& mi = *cx.mi;
  int item;
  if (leader) {
    item = atomicAdd(counter, 1);
    if (item > n_items) item = n_items;
    if (!C::PAIR) return item;
    WAIT2(&mi.item_free, free_par(p.item), W2_ITEM);      // the peer has read the previous one
    st_async_u32(map_to_cta(&mi.item, 1), static_cast<uint32_t>(item), map_to_cta(&mi.item_full, 1));
  } else {
    mbar_arrive_expect_tx(&mi.item_full, 4);
    if (!WAIT2(&mi.item_full, full_par(p.item), W2_ITEM)) return n_items;
    item = *reinterpret_cast<volatile int*>(&mi.item);
    mbar_arrive_remote(map_to_cta(&mi.item_free, 0));
  }
  ++p.item;
  return item;
}
// stage of the n-th use of the key ring (V: of the value ring), and how often the stage has been used before
template <class C, bool V>
__device__ __forceinline__ int stage_of(uint32_t n) { return V ? 2 * (n % C::NV) + (C::NV == C::NK) : 2 * (n % C::NK) + (C::NV != C::NK); }
template <class C, bool V>
__device__ __forceinline__ uint32_t lap_of(uint32_t n) { return n / (V ? C::NV : C::NK); }
// expects a stage's bytes over both CTAs on the leader's barrier of the ring's next stage; returns that barrier's address
// for the copies and the stage's place; 0 once a wait has run out (no copy is issued into a ring that nobody drains)
template <class C, bool V>
__device__ __forceinline__ uint32_t ring_stage(const Ctx2& cx, Prod& p, bool leader, uint8_t** dst) {
  Misc2& mi = *cx.mi;
  if (*cx.abort_flag) return 0;
  uint32_t& n = V ? p.v : p.k;
  const int s = stage_of<C, V>(n);
  if (!WAIT2(&mi.kv_free[s], free_par((lap_of<C, V>(n))), W2_KVFREE)) return 0;
  if (leader) mbar_arrive_expect_tx(&mi.kv_full[s], C::NCTA * C::STAGE_BYTES);
  *dst = cx.ring + s * C::STAGE_BYTES;
  ++n;
  return in_cta<C>(&mi.kv_full[s], 0);
}

// start of a kernel: barriers, tensor memory; every thread of the CTA calls
template <class C>
__device__ __forceinline__ void setup(Ctx2& cx, uint8_t* smem, int* status, int wait_kcycles, bool leader) {
  Misc2& mi = *reinterpret_cast<Misc2*>(smem + Off<C>::MISC);
  cx.mi = &mi;
  cx.sQ = smem + Off<C>::Q;
  cx.ring = smem + Off<C>::RING;
  cx.abort_flag = &mi.abort_flag;
  cx.status = status;
  if (threadIdx.x == 0) init_barriers2<C>(mi, wait_kcycles, leader);
  if (threadIdx.x / 32 == WARP_QK) { if constexpr (C::PAIR) tmem_alloc_pair(&mi.tmem_base, 512); else tmem_alloc(&mi.tmem_base, 512); }
  tc_fence_before_sync();
  __syncthreads();
  if constexpr (C::PAIR) cluster_sync_all();             // both CTAs' barriers exist before any remote arrive
  tc_fence_after_sync();
  cx.tmem = mi.tmem_base;
}

// end of a kernel: no CTA of a pair may exit while its peer can still signal it or read its shared memory
template <class C>
__device__ __forceinline__ void teardown(const Ctx2& cx) {
  tc_fence_before_sync();
  __syncthreads();
  if constexpr (C::PAIR) cluster_sync_all();
  if (threadIdx.x / 32 == WARP_QK) {
    // no tensor-core operation may still be running when its accumulators are freed: each issuer ended with a
    // commit to mma_done (an arrival in both CTAs of a pair).  Immediate in a clean run; after an abort this is what
    // makes the exit safe.  The wait ignores the abort flag and is bounded.
    mbar_wait_drain(&cx.mi->mma_done, 0, cx.abort_flag);
    tc_fence_after_sync();
    if constexpr (C::PAIR) tmem_dealloc_pair(cx.tmem, 512); else tmem_dealloc(cx.tmem, 512);
  }
}

// Producer, at the end: every copy issued must have landed before a CTA may exit.  In a run without a timed-out wait that
// follows from the last uses of the rings having been consumed (teardown waits for every tensor-core operation).  After
// an abort nothing is consumed any more: the leader, whose barriers count the bytes of both CTAs' copies, waits on
// them (ignoring the abort flag, bounded); its peer cannot observe the completion of its own last copies and lets a
// fixed pause pass that outlasts any copy in flight.
template <class C>
__device__ __forceinline__ void drain_copies(const Ctx2& cx, const Prod& p, bool leader) {
  Misc2& mi = *cx.mi;
  if (!*cx.abort_flag) return;
  if (leader) {
    for (uint32_t i = (p.k > C::NK ? p.k - C::NK : 0); i < p.k; ++i)
      mbar_wait_drain(&mi.kv_full[stage_of<C, false>(i)], full_par(lap_of<C, false>(i)), cx.abort_flag);
    for (uint32_t i = (p.v > C::NV ? p.v - C::NV : 0); i < p.v; ++i)
      mbar_wait_drain(&mi.kv_full[stage_of<C, true>(i)], full_par(lap_of<C, true>(i)), cx.abort_flag);
    for (uint32_t i = (p.q > C::NQ ? p.q - C::NQ : 0); i < p.q; ++i)
      mbar_wait_drain(&mi.q_full[i % C::NQ], full_par(i / C::NQ), cx.abort_flag);
  }
  abort_grace_pause(cx.abort_flag);
}

// ------------------------------------------------------------------ issuers (one elected thread each; of a pair: of the leader CTA)
// operand of the n-th use of a ring, once its copy has landed / the stage is free once what this thread has issued has run
template <class C, bool V>
__device__ __forceinline__ uint32_t wait_stage(const Ctx2& cx, uint32_t n) {
  const int s = stage_of<C, V>(n);
  WAIT2I(&cx.mi->kv_full[s], full_par((lap_of<C, V>(n))), W2_KVFULL);
  return smem_u32(cx.ring) + s * C::STAGE_BYTES;
}
template <class C, bool V>
__device__ __forceinline__ void free_stage(const Ctx2& cx, uint32_t n) { commit<C>(&cx.mi->kv_free[stage_of<C, V>(n)]); }

template <class C>
struct IssuerQK {
  const Ctx2& cx;
  uint32_t nd = 0, k = 0, nq = 0, ns = 0;                            // descriptors, key ring, query slots; uses of S, modulo 2 in bits
  uint32_t qa[2] = {0, 0};                                           // query operands of the two blocks in work
  __device__ __forceinline__ explicit IssuerQK(const Ctx2& c) : cx(c) {}
  __device__ __forceinline__ uint32_t wait_q() {
    WAIT2I(&cx.mi->q_full[nq % C::NQ], full_par(nq / C::NQ), W2_QFULL);
    const uint32_t q = smem_u32(cx.sQ) + (nq % C::NQ) * C::Q_BYTES;
    ++nq;
    return q;
  }
  __device__ __forceinline__ uint32_t wait_k() { return wait_stage<C, false>(cx, k); }
  __device__ __forceinline__ void free_k() { free_stage<C, false>(cx, k++); }
  // S = Q K^T for block b, once the S before it is in registers
  __device__ __forceinline__ void qk(int b, uint32_t k_smem) {
    constexpr uint32_t idesc = make_idesc_bf16_f32(TILE * C::NCTA, TILE, false, false);
    const uint32_t q_smem = b ? qa[1] : qa[0];
    const int sb = C::TWO_S ? b : 0;
    WAIT2I(&cx.mi->s_read[sb], free_par(ns >> sb), W2_SREAD);
    ns ^= 1u << sb;
    tc_fence_after_sync();
    if constexpr (C::PAIR) mma_ss_pair_k128<true>(cx.tmem + C::tm_s(b), q_smem, k_smem, idesc);
    else if constexpr (C::D == 128) mma_ss_k128(cx.tmem + C::tm_s(b), q_smem, k_smem, idesc);
    else mma_ss_k64(cx.tmem + C::tm_s(b), q_smem, k_smem, idesc);
    commit<C>(&cx.mi->s_full[b]);
  }
};

template <class C>
struct IssuerPV {
  const Ctx2& cx;
  uint32_t nd = 0, v = 0, tiles = 0, blocks = 0;                     // descriptors, value ring; tiles and blocks so far, modulo 2 in bit b
  __device__ __forceinline__ explicit IssuerPV(const Ctx2& c) : cx(c) {}
  __device__ __forceinline__ void free_v() { free_stage<C, true>(cx, v++); }
  // the accumulator of the block before has been read out
  __device__ __forceinline__ void wait_read_out(int b) { WAIT2I(&cx.mi->o_free[b], free_par(blocks >> b), W2_OFREE); }
  // O of block b += P V of the values next in the ring, in two halves as P arrives.  The values are waited for after P: by then
  // every earlier use of their stage is known to have landed (of a pair the other issuer takes sweep tiles through this ring).
  __device__ __forceinline__ void pv(int b, bool first, bool last) {
    Misc2& mi = *cx.mi;
    constexpr uint32_t idesc = make_idesc_bf16_f32(TILE * C::NCTA, C::D, false, true);
    const uint32_t tO = cx.tmem + C::TM_O + b * C::D, tP = cx.tmem + C::TM_P + b * 64;
    if (first) { wait_read_out(b); blocks ^= 1u << b; }
    const uint32_t par = full_par(tiles >> b);
    tiles ^= 1u << b;
    WAIT2I(&mi.p_half[b], par, W2_PHALF);                                            // keys 0..63 of P
    const uint32_t v_smem = wait_stage<C, true>(cx, v);
    tc_fence_after_sync();
    mma_ts_k64<C::PAIR>(tO, tP, v_smem, idesc, !first);
    WAIT2I(&mi.p_full[b], par, W2_PFULL);
    tc_fence_after_sync();
    mma_ts_k64<C::PAIR>(tO, tP + 32, v_smem + 8192, idesc, true);
    commit<C>(&mi.pv_done[b]);
    if (last) commit<C>(&mi.o_full[b]);
  }
};

// ------------------------------------------------------------------ softmax warps: hooks of softmax_tile for block b
template <class C>
struct Hooks {
  const Ctx2& cx;
  uint32_t p_half, p_full, s_read;                           // barriers (of the leader CTA)
  uint64_t* pv_done;
  uint32_t tiles;                                            // tiles of this block before the present one
  __device__ __forceinline__ Hooks(const Ctx2& c, int b)
      : cx(c), p_half(in_cta<C>(&c.mi->p_half[b], 0)), p_full(in_cta<C>(&c.mi->p_full[b], 0)),
        s_read(in_cta<C>(&c.mi->s_read[C::TWO_S ? b : 0], 0)), pv_done(&c.mi->pv_done[b]), tiles(0) {}
  __device__ __forceinline__ void on_read() const { warp_arrive_leader(s_read); }
  __device__ __forceinline__ void before_p() const { WAIT2S(pv_done, free_par(tiles), W2_PV); tc_fence_after_sync(); }
  __device__ __forceinline__ void on_half() const { warp_arrive_leader(p_half); }
  __device__ __forceinline__ void on_full() const { warp_arrive_leader(p_full); }
};

}  // namespace flash
}  // namespace pc
