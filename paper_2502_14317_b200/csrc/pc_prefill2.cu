// Chunk-local causal attention with fused query-window scores (Eq. 1-2, Eq. 5-6).
//
// A CTA owns TWO 128-row query blocks A and B that walk the same K/V tiles; while the softmax of one block runs the
// tensor cores work for the other.
//
// Head size 128 runs on CTA pairs (cluster of two, tcgen05 cta_group::2): four blocks share the tiles, every
// 128-key tile is split between the two shared memories (each CTA stages 64 keys of K and 64 head-dim columns of V) and
// one MMA of M = 256 feeds both SMs.  A single CTA's 128 x 128 x 128 product reads 128 bytes a cycle, all that shared
// memory gives; on a pair it reads 96, and the L2 traffic is halved.
// Head size 64 runs on single CTAs: its products are half as long, and the softmax is what bounds it.
//
// Roles, rings, barriers and the tensor memory: pc_flash.cuh.
//
// What bounds it: the board's power cap (1000 W) in any loop of these calls, so energy a tile, and beside it the MUFU pipe: a
// step (a key tile for both blocks of a CTA) takes some 2700 cycles, of which the exponentials keep that pipe busy for 2048, the
// products the tensor cores as long (head size 64: half as long); at any time at least one block is at its exponentials, but a
// warp alone does not fill the pipe.  Head size 128, in a loop, whole call, with an S of each block under P (3300 cycles a step)
// -> with one S for both in turn: 128K tokens in chunks of 8192, 32/8 heads 8.39 -> 7.89 ms; 32/32 heads, chunks of 4096
// 5.49 -> 5.31 ms; 24/8 heads, ragged 1.39 -> 1.33 ms.  Two issuing warps, and head size 64: figures in pc_flash.cuh.
// A third build, head size 128 on single CTAs, takes short chunks of odd groups (launch_prefill_t).
//
// Window scores: the unit that runs the last query tiles of a (chunk, kv-head) group then sweeps the keys once more
// with the transposed product K_j Qw^T (the CTAs of a pair take alternate key tiles; keys on TMEM lanes, window
// rows on columns), so Eq. 6 is a per-thread sum in a fixed order: deterministic, fp32, no atomics.
#include "pc_attn.h"
#include "pc_kernels.h"
#include "pc_flash.cuh"

namespace pc {

namespace {

using namespace flash;
// ------------------------------------------------------------------ work decomposition
// Groups = (chunk, kv-head).  A unit is what the blocks (four of a pair, two of a single CTA) take at a time.  Pair:
//   G % 4 == 0   one query tile of four q-heads (block A: heads 0, 1 of the four; B: heads 2, 3; one per CTA)
//   G % 2 == 0   two adjacent tiles of two q-heads (A: lower tile; B: upper tile; one head per CTA)
//   G odd        four adjacent tiles of one q-head (A: the lower two, B: the upper two; one per CTA; the lower tile of a
//                block walks one fully masked key tile, 3 % of the tiles at 32 tiles a chunk)
// single CTA: one tile of two q-heads, or (G odd) two adjacent tiles of one;
// counted from the last tile of the chunk.  Item 0 of a group (the tail item) holds the units with window rows for all
// q-heads, then the score sweep; the other items are one unit each, heaviest first.
// Items are dealt out in batches of groups whose keys and values stay in L2 together, heaviest first over the whole
// batch, so that what is dealt last is light (one group at a time, the last blocks ended 4 % after the median one).
// Few groups (SPREAD, a build of its own: the other's code stays as it is): a tail item would outlast everything else (d = 64, G = 4: two units and as many sweep steps as a
// unit has tiles, on one CTA), so every unit is an item, and the sweeps follow as items of their own, each over a slice of
// the keys.  A sweep waits until the blocks with the group's window rows, wherever they run, have counted themselves
// done: all of them were dealt out before the first sweep, and no unit waits for a sweep.
// With per-chunk lengths the query tiles of a shorter chunk are numbered from the END: slot v of the static
// decomposition (v = T - 1 is the last tile of a full-length chunk) is tile v - (T - T_c) of a chunk with T_c tiles.
// The window then always sits in the last one or two slots, which the tail item owns together with the score sweep.
struct Sched2 {
  int T, G, hpu, tpu, P, U, ntu, ipg, batch, hp, n_pass, wp;
};
template <class C, bool SPREAD>
__device__ __forceinline__ Sched2 make_sched2(const PrefillParams& p) {
  Sched2 s;
  s.T = (p.L + TILE - 1) / TILE;
  s.G = p.Hq / p.Hkv;
  constexpr int BLOCKS = 2 * C::NCTA;
  s.hpu = s.G % BLOCKS == 0 ? BLOCKS : (s.G % 2 == 0 ? 2 : 1);      // q-heads and tiles of a unit
  s.tpu = BLOCKS / s.hpu;
  s.P = s.G / s.hpu;
  s.U = (s.T + s.tpu - 1) / s.tpu;
  // tail units: those that can hold window rows (with per-chunk lengths the window of some chunk may straddle two
  // tiles even where that of a full-length chunk does not)
  const int ntt = (p.chunk_len != nullptr) ? (p.w > 1 ? 2 : 1) : s.T - (p.L - p.w) / TILE;
  s.ntu = (ntt + s.tpu - 1) / s.tpu;
  if (s.ntu > s.U) s.ntu = s.U;
  s.ipg = SPREAD ? s.U * s.P : 1 + (s.U - s.ntu) * s.P;
  const long long kv_bytes = (long long)p.L * (4 * C::D);    // K and V of a group
  s.batch = (int)((48ll << 20) / kv_bytes);
  if (s.batch < 1) s.batch = 1;
  s.wp = (p.w + 7) & ~7;                                  // window rows of a head in the sweep operand (multiple of 8)
  const int cap = TILE / s.wp, want = (s.G + 1) / 2;
  s.hp = cap < want ? cap : want;                         // window heads per CTA and sweep pass
  s.n_pass = (s.G + 2 * s.hp - 1) / (2 * s.hp);
  return s;
}
// item -> (group, item within the group)
__device__ __forceinline__ void decode_item(const Sched2& s, int n_groups, int item, int& group, int& within) {
  const int per_batch = s.batch * s.ipg;
  const int b = item / per_batch, rem = item - b * per_batch, g0 = b * s.batch;
  const int size = n_groups - g0 < s.batch ? n_groups - g0 : s.batch;
  within = rem / size;
  group = g0 + rem - within * size;
}
// length of chunk c in tokens (window included), clamped to (w, L]
__device__ __forceinline__ int chunk_length(const PrefillParams& p, int c) {
  if (p.chunk_len == nullptr) return p.L;
  int len = __ldg(p.chunk_len + c);
  len = len > p.L ? p.L : len;
  return len <= p.w ? p.w + 1 : len;
}
// blocks of unit x of a group, counted from the last tile of the chunk
template <class C>
__device__ __forceinline__ void decode_unit(const Sched2& s, int rank, int hkv, int x, Desc& d) {
  const int unit = x / s.P, set = x - unit * s.P;
  const int hi = s.T - 1 - unit * s.tpu - (s.T - (d.len + TILE - 1) / TILE);      // upper tile of the unit
  const int h0 = hkv * s.G + set * s.hpu;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    int top;                                              // upper tile of the block over both CTAs
    if (!C::PAIR) {
      d.h[b] = s.hpu == 2 ? h0 + b : h0;
      top = s.hpu == 2 ? hi : hi - 1 + b;
      d.t[b] = top;
    } else if (s.hpu == 4) { d.h[b] = h0 + 2 * b + rank; top = hi; d.t[b] = hi; }
    else if (s.hpu == 2) { d.h[b] = h0 + rank; top = hi - 1 + b; d.t[b] = top; }
    else { d.h[b] = h0; top = hi - 2 + 2 * b; d.t[b] = top - 1 + rank; }
    d.n[b] = top < 0 ? 0 : top + 1;
  }
}

}  // namespace

// ====================================================================================
//                                   KERNEL
// ====================================================================================
// tensor maps (boxes of 64 d): tm_q (128 tokens), tm_kh (rotated keys, 64 tokens), tm_k (rotated keys, 128 tokens), tm_v
// (128 tokens), tm_o (store, 128 tokens), tm_qw (wp tokens)
template <int D, bool PAIR, bool SPREAD>
__global__ void __launch_bounds__(NT2, 1)
prefill_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kh,
               const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
               const __grid_constant__ CUtensorMap tm_o, const __grid_constant__ CUtensorMap tm_qw,
               const __grid_constant__ PrefillParams prm) {
  using C = Cfg<D, PAIR>;
  constexpr int NCTA = C::NCTA, Q_BYTES = C::Q_BYTES, NQ = C::NQ;
  constexpr int TILE_STAGES = TILE * D * 2 / C::STAGE_BYTES, STAGE_ATOMS = C::ATOMS / TILE_STAGES;   // of a full key tile (score sweep)
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0;
  const bool leader = (rank == 0);
  if (tid == WARP_PRODUCER * 32) {
    tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_kh); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v);
    tma_prefetch_desc(&tm_qw);
  }
  Ctx2 cx;
  setup<C>(cx, smem, prm.status, prm.wait_kcycles, leader);
  Misc2& mi = *cx.mi;
  chain();

  if (warp >= WARP_PRODUCER) {
    setmaxnreg_dec<REGS_PREFILL.service>();
    if (warp == WARP_PRODUCER) {
      // ================================================================ TMA producer (both CTAs of a pair)
      if (elect_one()) {
        const Sched2 sch = make_sched2<C, SPREAD>(prm);
        const int n_groups = prm.C * prm.Hkv, n_unit_items = n_groups * sch.ipg, slices = SPREAD ? prm.sweep_slices : 1;
        const int n_items = n_unit_items + (SPREAD ? n_groups * slices : 0);
        const int rows_half = sch.hp * sch.wp;           // sweep operand rows per CTA and pass (B operand half)
        Prod p;
        // Once a wait has run out (abort flag) no new work is started: every role leaves its loops at the next
        // descriptor, this one also at the next tile, so that no copy is issued into a ring that nobody drains.
        while (!*cx.abort_flag) {
          const int item = next_item<C>(cx, p, leader, prm.counter, n_items);
          if (item >= n_items) break;
          int group, within;
          const bool unit_item = !SPREAD || item < n_unit_items;
          if (unit_item) decode_item(sch, n_groups, item, group, within);
          else { within = (item - n_unit_items) / n_groups; group = item - n_unit_items - within * n_groups; }      // within: slice
          Desc d;
          d.c = group / prm.Hkv;
          d.hkv = group - d.c * prm.Hkv;
          d.len = chunk_length(prm, d.c);
          uint8_t* dst;
          const bool tail = !SPREAD && within == 0;
          const int first = SPREAD ? within : (tail ? 0 : sch.ntu * sch.P + within - 1);
          const int nsub = tail ? sch.ntu * sch.P : (unit_item ? 1 : 0);
          for (int sub = 0; sub < nsub; ++sub) {
            d.kind = KIND_FLASH;
            decode_unit<C>(sch, rank, d.hkv, first + sub, d);
            if (d.n[1] == 0) continue;                    // (n[0] <= n[1])
            publish<C>(cx, p, d);
            for (int b = 0; b < 2; ++b) {
              if (d.n[b] == 0) continue;
              const int qs = p.q % NQ;
              WAIT2(&mi.q_free[qs], free_par(p.q / NQ), W2_QFREE);
              if (leader) mbar_arrive_expect_tx(&mi.q_full[qs], NCTA * Q_BYTES);
              const uint32_t bar = in_cta<C>(&mi.q_full[qs], 0);
              for (int a = 0; a < C::ATOMS; ++a)
                load_box<C>(cx.sQ + qs * Q_BYTES + a * 16384, &tm_q, bar, a * 64, d.h[b], d.t[b] * TILE, d.c);
              ++p.q;
            }
            for (int j = 0; j < d.n[1]; ++j) {
              const uint32_t kbar = ring_stage<C, false>(cx, p, leader, &dst);
              if (kbar) {
                if constexpr (PAIR)
                  for (int a = 0; a < 2; ++a) load_box<C>(dst + a * 8192, &tm_kh, kbar, a * 64, d.hkv, j * TILE + (int)rank * 64, d.c);
                else
                  for (int a = 0; a < C::ATOMS; ++a) load_box<C>(dst + a * 16384, &tm_k, kbar, a * 64, d.hkv, j * TILE, d.c);
              }
              const uint32_t vbar = ring_stage<C, true>(cx, p, leader, &dst);
              if (vbar)
                for (int a = 0; a < (PAIR ? 1 : C::ATOMS); ++a)
                  load_box<C>(dst + a * 16384, &tm_v, vbar, PAIR ? (int)rank * 64 : a * 64, d.hkv, j * TILE, d.c);
            }
          }
          if (tail || !unit_item) {
            // ---- score sweep: window queries of hp heads per CTA and pass, then this CTA's key tiles.  A head's rows
            // in the operand are the wp tokens that end with the chunk (wp = w rounded up to 8: the first wp - w rows
            // are not window rows and are left out of the sums; a start before token 0 reads zeros)
            const int all_steps = ((d.len + TILE - 1) / TILE + NCTA - 1) / NCTA;
            const int step0 = unit_item ? 0 : all_steps * within / slices;
            const int n_steps = (unit_item ? all_steps : all_steps * (within + 1) / slices) - step0;
            if (SPREAD) { d.t[0] = step0; d.t[1] = n_steps; }
            for (int u = 0; u < sch.n_pass && (!SPREAD || n_steps > 0); ++u) {
              d.kind = KIND_SWEEP;
              d.h[0] = u;
              publish<C>(cx, p, d);
              for (int b = 0; b < 3 - NCTA; ++b) {        // a pair's CTAs load a column half each, a single CTA both
                const int qs = p.q % NQ;
                WAIT2(&mi.q_free[qs], free_par(p.q / NQ), W2_QFREE);
                if (leader) mbar_arrive_expect_tx(&mi.q_full[qs], NCTA * rows_half * D * 2);
                const uint32_t bar = in_cta<C>(&mi.q_full[qs], 0);
                for (int i = 0; i < sch.hp; ++i) {
                  int g = u * 2 * sch.hp + ((int)rank + b) * sch.hp + i;
                  if (g >= sch.G) g = sch.G - 1;          // filler rows: loaded, never summed
                  for (int a = 0; a < C::ATOMS; ++a)
                    load_box<C>(cx.sQ + qs * Q_BYTES + a * 16384 + i * sch.wp * 128, &tm_qw, bar, a * 64, d.hkv * sch.G + g,
                                d.len - sch.wp, d.c);
                }
                ++p.q;
              }
              // a full key tile takes a stage of the key ring, of a pair also the one of the value ring that follows it in memory
              // (everything uses a pair's rings in step)
              for (int jj = 0; jj < n_steps; ++jj)
                for (int i = 0; i < TILE_STAGES; ++i) {
                  const uint32_t kbar = i == 0 ? ring_stage<C, false>(cx, p, leader, &dst) : ring_stage<C, true>(cx, p, leader, &dst);
                  if (kbar)
                    for (int a = 0; a < STAGE_ATOMS; ++a)
                      load_box<C>(dst + a * 16384, &tm_k, kbar, (i * STAGE_ATOMS + a) * 64, d.hkv, (NCTA * (step0 + jj) + (int)rank) * TILE, d.c);
                }
            }
          }
        }
        Desc d;
        d.kind = KIND_DONE; d.c = d.hkv = d.len = 0;
        publish<C>(cx, p, d, D == 128 || prm.skip_final_publication == 0);
        drain_copies<C>(cx, p, leader);
      }
      __syncwarp();
    } else if (warp == WARP_QK && leader) {
      // ================================================================ issuer of Q K^T (of a pair: leader CTA)
      if (elect_one()) {
        const Sched2 sch = make_sched2<C, SPREAD>(prm);
        const int rows_half = sch.hp * sch.wp;
        const uint32_t idesc_sw = make_idesc_bf16_f32(TILE * NCTA, PAIR ? 2 * rows_half : (rows_half + 15) & ~15, false, false);
        IssuerQK<C> is(cx);
        uint32_t nt = 0, n_go = 0;
        bool flashed = false;                                    // a unit since the last sweep: both issuers agree on it
        while (true) {
          const Desc d = next_desc<C>(cx, is.nd, false);
          if (d.kind == KIND_DONE) break;
          if (d.kind == KIND_FLASH) {
            flashed = true;
            // The blocks take turns on S.  One copy of a product each here and below, whatever block takes it (pc_parallel.cu):
            // us in loops of 15 ms, copies for the two blocks / one, head size 64, 8 chunks of 4096, 32/8 heads 914 / 860, 22 of 958 278 / 257; head
            // size 128, 8 of 8192, 32/8 heads 4017 / 3962, 8 of 4096, 32/32 heads 1375 / 1334, 4 of 1257 134 / 128; of Q K^T alone:
            // nothing, of P V alone: half of it.  In long loops, at the power cap, two thirds of that.
            for (int j = 0; j < d.n[1]; ++j) {
              const uint32_t k_u32 = is.wait_k();
#pragma unroll 1
              for (int b = j < d.n[0] ? 0 : 1; b < 2; ++b) {
                if (j == 0) { const uint32_t q = is.wait_q(); if (b) is.qa[1] = q; else is.qa[0] = q; }
                is.qk(b, k_u32);
              }
              is.free_k();
            }
          } else {
            // ---- score sweep, one pass: S^T = K_j Qw^T.  Its two [128 keys x 256 rows] buffers overlay all of TMEM:
            // every S / P buffer is consumed and the accumulators have been read out.
            const int n_steps = SPREAD ? d.t[1] : ((d.len + TILE - 1) / TILE + NCTA - 1) / NCTA;
            if (flashed) { WAIT2S(&mi.sweep_go, full_par(n_go), W2_SWEEP); ++n_go; }
            flashed = false;
            for (int b = 0; b < 3 - NCTA; ++b) is.qa[b] = is.wait_q();
            for (int jj = 0; jj < n_steps; ++jj, ++nt) {
              const int e = nt & 1;
              WAIT2S(&mi.t_free[e], free_par(nt >> 1), W2_TFREE);
              const uint32_t k_u32 = is.wait_k();
              if constexpr (PAIR) {
                wait_stage<C, true>(cx, is.k);                   // (the rings are in step)
                tc_fence_after_sync();
                mma_ss_pair_k128<false>(cx.tmem + e * 256, k_u32, is.qa[0], idesc_sw);
              } else {
                tc_fence_after_sync();
                for (int b = 0; b < 2; ++b) {
                  if constexpr (D == 128) mma_ss_k128(cx.tmem + e * 256 + b * 128, k_u32, is.qa[b], idesc_sw);
                  else mma_ss_k64(cx.tmem + e * 256 + b * 128, k_u32, is.qa[b], idesc_sw);
                }
              }
              commit<C>(&mi.t_full[e]);
              if constexpr (PAIR) free_stage<C, true>(cx, is.k);
              is.free_k();
            }
            // what follows overwrites the sweep buffers: wait until both were read
            WAIT2S(&mi.t_free[nt & 1], free_par(nt >> 1), W2_TFREE);
            WAIT2S(&mi.t_free[(nt + 1) & 1], free_par((nt + 1) >> 1), W2_TFREE);
          }
        }
        commit<C>(&mi.mma_done);                                 // teardown waits for everything the issuers issued
      }
      __syncwarp();
    } else if (warp == WARP_PV && leader) {
      // ================================================================ issuer of P V (of a pair: leader CTA)
      if (elect_one()) {
        IssuerPV<C> is(cx);
        bool flashed = false;
        while (true) {
          const Desc d = next_desc<C>(cx, is.nd, false);
          if (d.kind == KIND_DONE) break;
          if (d.kind == KIND_FLASH) {
            flashed = true;
            for (int j = 0; j < d.n[1]; ++j) {
#pragma unroll 1
              for (int b = j < d.n[0] ? 0 : 1; b < 2; ++b) is.pv(b, j == 0, j == (b ? d.n[1] : d.n[0]) - 1);
              is.free_v();
            }
          } else {
            // (one signal per run of sweeps: with one per sweep this thread could be two phases ahead of the one that waits)
            if (flashed) {
              for (int b = 0; b < 2; ++b) is.wait_read_out(b);
              tc_fence_after_sync();
              tc_fence_before_sync();
              mbar_arrive(&mi.sweep_go);
            }
            flashed = false;
            if (PAIR) is.v += SPREAD ? d.t[1] : ((d.len + TILE - 1) / TILE + NCTA - 1) / NCTA;
          }
        }
        commit<C>(&mi.mma_done);
      }
      __syncwarp();
    }
  } else if (warp >= WARP_EPI) {
    // ================================================================ epilogue: normalise, stage bf16 rows in the block's
    // (now idle) query slot, TMA store
    setmaxnreg_dec<REGS_PREFILL.epilogue>();
    const Sched2 sch = make_sched2<C, SPREAD>(prm);
    const int r = tid & 127;
    const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
    uint32_t nd = 0, nq = 0, no[2] = {0, 0};
    while (true) {
      const Desc d = next_desc<C>(cx, nd, true);
      if (d.kind == KIND_DONE) break;
      if (d.kind == KIND_SWEEP) {
        if (!SPREAD && d.h[0] == 0) {                            // the window rows' log-sum-exp of this CTA's blocks is in memory
          __threadfence();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive_cluster(in_cta<C>(&mi.lse_rdy, 0));
            if (PAIR) mbar_arrive_cluster(in_cta<C>(&mi.lse_rdy, 1));
          }
        }
        nq += 3 - NCTA;
        continue;
      }
#pragma unroll 1
      for (int b = 0; b < 2; ++b) {
        if ((b ? d.n[1] : d.n[0]) == 0) continue;
        const int h = b ? d.h[1] : d.h[0], t = b ? d.t[1] : d.t[0];
        const uint32_t ph = b ? no[1]++ : no[0]++;
        uint8_t* const myQ = cx.sQ + (nq % NQ) * Q_BYTES;
        uint64_t* const q_free = &mi.q_free[nq % NQ];
        ++nq;
        const int token = t * TILE + r;
        WAIT2(&mi.lm_full[b], full_par(ph), W2_LM);
        const float m_used = mi.lm[b][0][r], l_run = mi.lm[b][1][r];
        warp_arrive(&mi.lm_free[b]);
        WAIT2S(&mi.o_full[b], full_par(ph), W2_OFULL);
        tc_fence_after_sync();
        const bool in_chunk = token >= 0 && token < d.len;       // rows behind the end of the chunk are written as zeros
        const float inv_l = in_chunk ? 1.0f / l_run : 0.0f;
        const uint32_t tO = cx.tmem + C::TM_O + b * D + lane_sel;
#pragma unroll 1
        for (int q = 0; q < D / 32; ++q) {
          uint32_t o[32];
          tmem_ld32(tO + q * 32, o);
          tmem_wait_ld();
          loaded(o);
#pragma unroll
          for (int g4 = 0; g4 < 4; ++g4) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              pk[e] = in_chunk ? pack_bf16x2(__uint_as_float(o[g4 * 8 + 2 * e]) * inv_l, __uint_as_float(o[g4 * 8 + 2 * e + 1]) * inv_l) : 0u;
            const int col = q * 32 + g4 * 8;
            *reinterpret_cast<uint4*>(myQ + (col / 64) * 16384 + sw128_offset(r, (col % 64) / 8)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
        warp_arrive_leader(in_cta<C>(&mi.o_free[b], 0));
        if (in_chunk) {
          const float lse2 = m_used + log2f(l_run);
          const size_t row = (size_t)d.c * prm.Hq + h;
          if (prm.lse) prm.lse[row * prm.L + token] = lse2 * 0.6931471805599453f;
          const int wi = token - (d.len - prm.w);
          if (wi >= 0) {
            prm.win_lse2[row * prm.w + wi] = lse2;               // for the score sweep
            if (prm.win_lse != nullptr) prm.win_lse[row * prm.w + wi] = lse2 * 0.6931471805599453f;
          }
        }
        fence_proxy_async_smem();
        named_barrier_sync(1, 128);
        if (SPREAD && r == 0 && (t + 1) * TILE > d.len - prm.w && t * TILE < d.len) {     // a block with window rows
          __threadfence();
          atomicAdd(prm.counter + 1 + d.c * prm.Hkv + d.hkv, 1);
        }
        if (r == 0) {
          if (t >= 0 && t * TILE < prm.L) {
            for (int a = 0; a < C::ATOMS; ++a) tma_store_4d(&tm_o, myQ + a * 16384, a * 64, h, t * TILE, d.c);
            tma_store_commit();
            tma_store_wait_read();
          }
          mbar_arrive(q_free);
        }
      }
    }
    leave_group<4>(1, (no[0] + no[1]) & 1u, &mi.left[0]);        // (a meeting per block)
    if (r == 0) tma_store_wait_all();
  } else {
    // ================================================================ softmax
    setmaxnreg_inc<REGS_PREFILL.softmax>();
    const Sched2 sch = make_sched2<C, SPREAD>(prm);
    const int b = warp >> 2;
    const int r = tid & 127;
    const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tS = cx.tmem + C::tm_s(b) + lane_sel, tP = cx.tmem + C::TM_P + b * 64 + lane_sel;
    const uint32_t tO = cx.tmem + C::TM_O + b * D + lane_sel;
    const float scale_log2 = prm.scale_log2;
    Hooks<C> hk(cx, b);
    uint32_t nd = 0, n_s = 0, n_blk = 0, nq = 0, nt = 0, n_lse = 0;
    while (true) {
      const Desc d = next_desc<C>(cx, nd, true);
      if (d.kind == KIND_DONE) break;
      if (d.kind == KIND_FLASH) {
        nq += d.n[0] > 0 ? 2 : 1;
        const int n = b ? d.n[1] : d.n[0], t = b ? d.t[1] : d.t[0];
        if (n == 0) continue;
        RowState st = {-INFINITY, 0.0f};
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
          WAIT2S(&mi.s_full[b], full_par(n_s), W2_SFULL);
          ++n_s;
          tc_fence_after_sync();
          if (j > 0 && j < t) softmax_tile<D, false>(tS, tP, tO, TILE, false, scale_log2, st, hk);
          else softmax_tile<D, true>(tS, tP, tO, (t - j) * TILE + r + 1, j == 0, scale_log2, st, hk);   // causal: keys <= token
          ++hk.tiles;
        }
        WAIT2S(&mi.lm_free[b], free_par(n_blk), W2_LMFREE);
        ++n_blk;
        mi.lm[b][0][r] = st.m;
        mi.lm[b][1][r] = st.l;
        warp_arrive(&mi.lm_full[b]);
      } else {
        // ---- score sweep: this thread owns a key; its warpgroup sums the columns of the heads that CTA b loaded
        const int u = d.h[0];
        if (u == 0) {
          if constexpr (SPREAD) {
            // Sweeps follow one another here without a block between them, so the epilogue warps, which would be several sweeps
            // ahead, cannot hand this over through a barrier's parity.  The log-sum-exp of all the group's window rows is in
            // memory once its blocks have counted themselves done, and the epilogue has read this CTA's last
            // statistics (lm, reused below) once each warpgroup has seen its own lm_free.
            WAIT2S(&mi.lm_free[b], free_par(n_blk), W2_LMFREE);
            if (lane == 0) {
              const int tiles = (d.len + TILE - 1) / TILE - (d.len - prm.w) / TILE;
              wait_count(prm.counter + 1 + d.c * prm.Hkv + d.hkv, tiles * sch.G, cx.abort_flag, cx.status, C::CODE + W2_LSE);
            }
            named_barrier_sync(3, 256);
            ++n_lse;
          } else {
            mbar_wait_cluster(&mi.lse_rdy, full_par(n_lse), cx.abort_flag, cx.status, C::CODE + W2_LSE);
            ++n_lse;
          }
        }
        const int rows_half = sch.hp * sch.wp;
        const int g0 = u * 2 * sch.hp + b * sch.hp;
        const int heads = sch.G - g0 < sch.hp ? (sch.G > g0 ? sch.G - g0 : 0) : sch.hp;
        const int cols = heads * sch.wp;
        // log-sum-exp of the columns' window rows in log2 units; +inf (probability 0) in columns that are no window rows
        float* const lse_cols = &mi.lm[1][b][0];
        if (r < cols) {
          const int wi = r % sch.wp - (sch.wp - prm.w);
          float x = INFINITY;
          if (wi >= 0) x = __ldcg(prm.win_lse2 + ((size_t)d.c * prm.Hq + d.hkv * sch.G + g0 + r / sch.wp) * prm.w + wi);
          lse_cols[r] = x;
        }
        named_barrier_sync(3, 256);
        const int n_steps = SPREAD ? d.t[1] : ((d.len + TILE - 1) / TILE + NCTA - 1) / NCTA;
        const int w0 = d.len - prm.w, pad = sch.wp - prm.w;      // first window token of this chunk
        float* const xch = &mi.lm[0][0][0];                      // [buffer][key]
        const uint32_t t_free0 = in_cta<C>(&mi.t_free[0], 0), t_free1 = in_cta<C>(&mi.t_free[1], 0);
        for (int jj = 0; jj < n_steps; ++jj, ++nt) {
          const int e = nt & 1;
          WAIT2S(&mi.t_full[e], full_par(nt >> 1), W2_TFULL);
          tc_fence_after_sync();
          const int key0 = (NCTA * ((SPREAD ? d.t[0] : 0) + jj) + (int)rank) * TILE, key = key0 + r;
          const uint32_t tT = cx.tmem + e * 256 + b * (PAIR ? rows_half : 128) + lane_sel;
          float part = 0.0f;
          int col = 0;
          if (key0 + TILE - 1 <= w0) {                           // every window row sees every key of the tile
            const uint64_t scale2 = dup2(scale_log2);
            uint64_t sum2 = 0ull;
#pragma unroll 1
            for (; col + 32 <= cols; col += 32) {
              uint32_t sv[32];
              tmem_ld32(tT + col, sv);
              tmem_wait_ld();
              loaded(sv);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float4 l4 = *reinterpret_cast<const float4*>(lse_cols + col + (i / 2) * 4);
                const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(sv[2 * i]), __uint_as_float(sv[2 * i + 1])), scale2,
                                              (i & 1) ? pack_f32x2(-l4.z, -l4.w) : pack_f32x2(-l4.x, -l4.y));
                float x0, x1;
                unpack_f32x2(x2, x0, x1);
                sum2 = add_f32x2(sum2, pack_f32x2(fast_exp2(x0), fast_exp2(x1)));
              }
            }
            float a0, a1;
            unpack_f32x2(sum2, a0, a1);
            part = a0 + a1;
          }
#pragma unroll 1
          for (; col < cols; col += 8) {                         // the rest, and tiles that reach into the window
            uint32_t sv[8];
            tmem_ld8(tT + col, sv);
            const float4 la = *reinterpret_cast<const float4*>(lse_cols + col), lb = *reinterpret_cast<const float4*>(lse_cols + col + 4);
            const float ls[8] = {la.x, la.y, la.z, la.w, lb.x, lb.y, lb.z, lb.w};
            const int wi0 = col % sch.wp - pad;                  // window row of the first of these columns (negative: none)
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float pv = fast_exp2(fmaf(__uint_as_float(sv[i]), scale_log2, -ls[i]));
              part += key <= w0 + wi0 + i ? pv : 0.0f;
            }
          }
          warp_arrive_leader(e ? t_free1 : t_free0);
          if (b == 1) xch[e * TILE + r] = part;
          named_barrier_sync(3, 256);
          if (b == 0 && key < d.len) {
            float* dst = prm.win_score + ((size_t)d.c * prm.Hkv + d.hkv) * prm.L + key;
            const float total = part + xch[e * TILE + r];
            *dst = (u == 0) ? total : (*dst + total);
          }
        }
        named_barrier_sync(3, 256);                              // everyone is past the exchange buffer
        if (tid == 0)                                            // the window queries were read by MMAs that have completed
          for (int i = 0; i < 3 - NCTA; ++i) mbar_arrive(&mi.q_free[(nq + i) % NQ]);
        nq += 3 - NCTA;
      }
    }
    // (meetings of a sweep pass: one per step and two more, with SPREAD a third in the first pass)
    leave_group<8>(3, (nt + (SPREAD ? n_lse : 0u)) & 1u, &mi.left[1]);
  }

  teardown<C>(cx);
}

// ====================================================================================
//                                   host launcher
// ====================================================================================
// Slices of a group's score sweep as items of their own (SPREAD), or 0 for sweeps inside the tail items.  Where a tail item has more
// steps (tiles of its units and of the sweep) than 1.2 times what a CTA or pair gets on average: us without / with, C x L,
// heads, d: 1 x 2048, 32/8, 64 (3.1 times) 99 / 54; 1 x 8192, 16/4, 64 (1.7) 332 / 231; 2 x 1024, 8/2, 128 (5.5) 41.6 / 38.1;
// 2 x 2048, 32/8, 128 (0.8) 100 / 105; 3 x 3000, 24/8, 128 (1.0) 215 / 223.  Chunks of a few tiles only where the heads
// of a group are several units (1 x 206, 14/2, 64 44.0 / 20.9; 1 x 250, 32/8, 64 22.3 / 19.5; 4 x 300, 24/8, 128 43.7 / 38.0;
// 4 x 500, 28/4, 128 79 / 43): with one unit the count in memory costs more than it spreads (1 x 192, 32/8, 128 20.5 / 21.6;
// 8 x 512, 8/2, 128 31.5 / 33.3).
template <class C>
static int sweep_slices(const PrefillParams& p, int units) {
  constexpr int NCTA = C::NCTA, BLOCKS = 2 * NCTA;
  const long long groups = (long long)p.C * p.Hkv;
  const int T = (p.L + TILE - 1) / TILE;
  if (groups > MAX_SPREAD_GROUPS || T < 2) return 0;
  const int G = p.Hq / p.Hkv, hpu = G % BLOCKS == 0 ? BLOCKS : (G % 2 == 0 ? 2 : 1), tpu = BLOCKS / hpu;
  const int P = G / hpu, U = (T + tpu - 1) / tpu;
  if (P == 1 && T < 6) return 0;
  const int steps = (T + NCTA - 1) / NCTA;
  const double all = (double)groups * (P * U * (T + tpu) / 2.0 + steps), tail = (double)P * T + steps;
  if (tail < 1.2 * all / units) return 0;
  int n = (int)(units / groups) < 8 ? (int)(units / groups) : 8;
  n = n < steps ? n : steps;
  return n < 1 ? 1 : n;
}

template <int D, bool PAIR, bool SPREAD>
static cudaError_t launch_build(const CUtensorMap* maps, const PrefillParams& prm, int grid, cudaStream_t st) {
  // the opt-in to large dynamic shared memory is a per-device attribute of the function: set it on every call
  // (a host-side call of a few hundred nanoseconds) rather than remember which devices have it
  using C = Cfg<D, PAIR>;
  constexpr auto kernel = prefill_kernel<D, PAIR, SPREAD>;
  if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Off<C>::TOTAL); e != cudaSuccess) return e;
  return launch_chained(kernel, dim3((unsigned)grid), dim3(NT2), Off<C>::TOTAL, st, C::NCTA, maps[0], maps[5], maps[1], maps[2],
                        maps[3], maps[4], prm);
}
template <int D>
static cudaError_t launch_prefill_t(const CUtensorMap* maps, PrefillParams prm, int sm_count, cudaStream_t st) {
  using C = Cfg<D, D == 128>;
  const int grid = sm_count / C::NCTA * C::NCTA;         // one CTA per SM, a whole number of pairs
  if (grid < 1) return cudaErrorInvalidConfiguration;
  prm.sweep_slices = sweep_slices<C>(prm, grid / C::NCTA);
  // Odd G and chunks that do not fill a pair's unit of four tiles: single CTAs (two tiles) where there are more groups than pairs, so
  // that a group per CTA is not what counts.  us, pairs / single CTAs, C x L, heads, d = 128: 128 x 128, 32/32 508 / 314;
  // 32 x 256, 32/32 186 / 145; 128 x 256, 24/8 373 / 303; 128 x 300, 32/32 953 / 720; fewer groups: 12 x 256, 28/4 (48) 63 / 80.
  if constexpr (C::PAIR)
    if (prm.Hq / prm.Hkv % 2 != 0 && prm.L <= 3 * TILE && (long long)prm.C * prm.Hkv > grid / C::NCTA)
      return launch_build<D, false, false>(maps, prm, sm_count, st);
  return prm.sweep_slices > 0 ? launch_build<D, C::PAIR, true>(maps, prm, grid, st) : launch_build<D, C::PAIR, false>(maps, prm, grid, st);
}

__global__ void __launch_bounds__(256) win_lse_natural_kernel(float* x, long long n) {
  chain();
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) x[i] *= 0.6931471805599453f;
}
cudaError_t launch_win_lse_natural(float* x, long long n, cudaStream_t st) {
  return launch_chained(win_lse_natural_kernel, dim3((unsigned)((n + 255) / 256 < 1184 ? (n + 255) / 256 : 1184)), dim3(256), 0, st, 1, x, n);
}

// maps: 0 q (box 64 x 128 tokens), 1 rotated keys (64 x 128), 2 v (64 x 128), 3 o (store), 4 q with a
// wp-token box, 5 rotated keys with a 64-token box
cudaError_t launch_prefill_attn(const CUtensorMap* maps, const PrefillParams& prm, int d, int sm_count, cudaStream_t st) {
  return d == 128 ? launch_prefill_t<128>(maps, prm, sm_count, st) : launch_prefill_t<64>(maps, prm, sm_count, st);
}

}  // namespace pc
