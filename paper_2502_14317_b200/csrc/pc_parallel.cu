// Parallel (global) attention of the query window over the compressed cache (Sec. 3.1 "Global attention",
// Eq. 9-11): every shape with more than 32 query rows per kv-head (fewer: pc_decode.cu).
//
// Two query blocks per CTA with a softmax warpgroup each, roles and rings as in pc_flash.cuh.  Rows = the w window
// queries of the q-heads of one kv-head, head-major; they all read the same cache.  Two ways to fill the blocks:
//   alt = 1  both blocks hold the same rows and take alternate key tiles, each with its own maximum, sum and accumulator;
//            the epilogue adds them up.  128 rows per CTA, 256 per CTA pair (head size 128).
//   alt = 0  the blocks hold different rows and share every tile: 256 rows per CTA, 512 per pair.
// Head size 128 with more than 128 rows runs on CTA pairs (half the shared-memory operands and L2 traffic of two single
// CTAs), everything else on single CTAs.  An item is (sequence, kv-head, row group, key split); the last tile of the
// last split holds the window's own keys (causal by the row's window index), a ragged last cache tile is masked by
// count.  Queries arrive rotated.  Small batches split the keys; the splits' fp32 partial results are merged
// by a second kernel.
//
// What bounds it: many sequences, the power cap and the tile's softmax (2048 cycles a step on the MUFU pipe at the least): 64
// sequences of 64 queries over 16384 entries, 32/8 heads 1.23 -> 1.17 ms in a loop with one S for both blocks in turn
// (pc_flash.cuh).  Head size 128 with few rows: caches are read at 5 TB/s.  One sequence: latencies, half of the cycles in the
// tiles of an item, the rest writing its partial rows, cold code, setup and exit: 34.6 -> 33.0 us (with the rotation and the
// merge) with one S, 31.6 with two issuing warps, 30.2 with one copy of their code.
//
// The issuers' loops hold one copy of a product each, whatever block takes it.  With copies of their own for the two blocks
// every warp was slower; probably the instruction caches, which all warps share.  In a loop, us, one issuing thread / two with
// copies / two without: head size 64, window of 16 over 64 caches of 16000, 32/8 heads 449 / 513 / 446, window of 64 over one
// of 16384 28.6 / 30.2 / 27.9; head size 128, window of 64 over 64 caches of 16384, 32/8 heads 1140 / 1175 / 1107, over one
// 33.2 / 31.2 / 30.1.
#include "pc_attn.h"
#include "pc_flash.cuh"
#include "pc_kernels.h"

namespace pc {

namespace {

using namespace flash;

struct Item {
  int seq, hkv, rg, split, j0, n;              // key tiles j0 .. j0 + n - 1
};
__device__ __forceinline__ Item decode_item(const ParallelParams& p, int item) {
  Item it;
  it.split = item % p.n_split;
  int x = item / p.n_split;
  it.rg = x % p.n_rg; x /= p.n_rg;
  it.hkv = x % p.Hkv;
  it.seq = x / p.Hkv;
  const int n_all = p.n_cache_tiles + 1;
  it.j0 = (int)((long long)n_all * it.split / p.n_split);
  it.n = (int)((long long)n_all * (it.split + 1) / p.n_split) - it.j0;
  return it;
}

}  // namespace

// tensor maps (boxes of 64 d): tm_q (rotated window queries, one head, w tokens), tm_kc (cache keys, 64 of a pair or 128),
// tm_vc (cache values, 128), tm_kw (window keys, 64 or 128), tm_vw (window values, 128).  Rows of a box behind the end
// of the tensor read as zeros; the softmax masks those keys.
template <int D, bool PAIR>
__global__ void __launch_bounds__(NT2, 1)
parallel_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kc,
                     const __grid_constant__ CUtensorMap tm_vc, const __grid_constant__ CUtensorMap tm_kw,
                     const __grid_constant__ CUtensorMap tm_vw, const __grid_constant__ ParallelParams prm) {
  using C = Cfg<D, PAIR>;
  constexpr int NCTA = C::NCTA, NQ = C::NQ;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0;
  const bool leader = (rank == 0), alt = prm.alt != 0;
  const int w = prm.w, G = prm.Hq / prm.Hkv, hpb = TILE / w;                 // q-heads per 128-row block
  const int group_heads = hpb * NCTA * (alt ? 1 : 2);
  // first q-head (within the kv-head's G) of block b of CTA `r` in row group rg
  auto first_head = [&](int rg, int b, int r) { return rg * group_heads + ((alt ? 0 : b * NCTA) + r) * hpb; };
  if (G % group_heads != 0) {                                                // rows without a query: finite operands
    for (int i = tid; i < NQ * C::Q_BYTES / 16; i += NT2) reinterpret_cast<uint4*>(smem + Off<C>::Q)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  if (tid == WARP_PRODUCER * 32) { tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_kc); tma_prefetch_desc(&tm_vc); }
  Ctx2 cx;
  setup<C>(cx, smem, prm.status, prm.wait_kcycles, leader);
  Misc2& mi = *cx.mi;
  chain();

  if (warp >= WARP_PRODUCER) {
    setmaxnreg_dec<REGS_PARALLEL.service>();
    if (warp == WARP_PRODUCER) {
      // ================================================================ TMA producer (both CTAs of a pair)
      if (elect_one()) {
        const int n_items = prm.B * prm.Hkv * prm.n_rg * prm.n_split;
        Prod p;
        // once a wait has run out (abort flag) no new work is started
        while (!*cx.abort_flag) {
          const int item = next_item<C>(cx, p, leader, prm.counter, n_items);
          if (item >= n_items) break;
          const Item it = decode_item(prm, item);
          Desc d;
          d.kind = KIND_FLASH;
          d.c = it.seq; d.hkv = it.hkv; d.len = it.split;
          d.h[0] = it.rg; d.h[1] = 0;
          d.t[0] = it.j0; d.t[1] = it.n;
          d.n[0] = alt ? (it.n + 1) / 2 : it.n;
          d.n[1] = alt ? it.n / 2 : (first_head(it.rg, 1, 0) < G ? it.n : 0);
          publish<C>(cx, p, d);
          for (int b = 0; b < (alt ? 1 : 2); ++b) {
            if (d.n[b] == 0) continue;
            const int qs = p.q % NQ;
            WAIT2(&mi.q_free[qs], free_par(p.q / NQ), W2_QFREE);
            auto heads = [&](int r) {                                       // q-heads of the block in CTA r
              const int left = G - first_head(it.rg, b, r);
              return r >= NCTA || left < 0 ? 0 : (left < hpb ? left : hpb);
            };
            if (leader) mbar_arrive_expect_tx(&mi.q_full[qs], (heads(0) + heads(1)) * w * D * 2);
            const uint32_t bar = in_cta<C>(&mi.q_full[qs], 0);
            for (int i = 0; i < heads(rank); ++i)
              for (int a = 0; a < C::ATOMS; ++a)
                load_box<C>(cx.sQ + qs * C::Q_BYTES + a * 16384 + i * w * 128, &tm_q, bar, a * 64,
                            it.hkv * G + first_head(it.rg, b, rank) + i, 0, it.seq);
            ++p.q;
          }
          // order of the copies: K of the first tile (alt: of the first two), then V of tile t and the K that follows it in use
          uint8_t* dst;
          auto load_k = [&](int t) {
            const uint32_t bar = ring_stage<C, false>(cx, p, leader, &dst);
            if (!bar) return;
            const int j = it.j0 + t, key0 = PAIR ? (int)rank * 64 : 0;
            for (int a = 0; a < C::ATOMS; ++a) {
              uint8_t* const to = dst + a * (PAIR ? 8192 : 16384);
              if (j < prm.n_cache_tiles) load_box<C>(to, &tm_kc, bar, a * 64, j * TILE + key0, it.hkv, it.seq);
              else load_box<C>(to, &tm_kw, bar, a * 64, it.hkv, key0, it.seq);
            }
          };
          const int lag = alt ? 2 : 1;
          for (int t = 0; t < lag && t < it.n; ++t) load_k(t);
          for (int t = 0; t < it.n; ++t) {
            const uint32_t bar = ring_stage<C, true>(cx, p, leader, &dst);
            const int j = it.j0 + t;
            if (bar)
              for (int a = 0; a < (PAIR ? 1 : C::ATOMS); ++a) {
                const int col = PAIR ? (int)rank * 64 : a * 64;
                if (j < prm.n_cache_tiles) load_box<C>(dst + a * 16384, &tm_vc, bar, col, j * TILE, it.hkv, it.seq);
                else load_box<C>(dst + a * 16384, &tm_vw, bar, col, it.hkv, 0, it.seq);
              }
            if (t + lag < it.n) load_k(t + lag);
          }
        }
        Desc d;
        d.kind = KIND_DONE; d.c = d.hkv = d.len = 0;
        publish<C>(cx, p, d, prm.skip_final_publication == 0);
        // test hook: nobody takes the message, so this wait runs out as the consumers' do, and the copies are drained as after
        // any abort
        if (prm.skip_final_publication != 0) WAIT2(&mi.d_free[(p.d - 1) % NDESC], free_par((p.d - 1) / NDESC + 1), W2_DESC);
        drain_copies<C>(cx, p, leader);
      }
      __syncwarp();
    } else if (warp == WARP_QK && leader) {
      // ================================================================ issuer of Q K^T (of a pair: leader CTA)
      if (elect_one()) {
        IssuerQK<C> is(cx);
        while (true) {
          const Desc d = next_desc<C>(cx, is.nd, false);
          if (d.kind == KIND_DONE) break;
          const int n = d.t[1];
          is.qa[0] = is.qa[1] = is.wait_q();
          if (!alt && d.n[1] > 0) is.qa[1] = is.wait_q();
          for (int t = 0; t < n; ++t) {
            const uint32_t k_u32 = is.wait_k();
            const int first = alt ? t & 1 : 0, last = alt ? first : (d.n[1] > 0 ? 1 : 0);       // blocks that take the tile
#pragma unroll 1
            for (int b = first; b <= last; ++b) is.qk(b, k_u32);
            is.free_k();
          }
        }
        commit<C>(&mi.mma_done);                                             // teardown waits for everything the issuers issued
      }
      __syncwarp();
    } else if (warp == WARP_PV && leader) {
      // ================================================================ issuer of P V (of a pair: leader CTA)
      if (elect_one()) {
        IssuerPV<C> is(cx);
        while (true) {
          const Desc d = next_desc<C>(cx, is.nd, false);
          if (d.kind == KIND_DONE) break;
          const int n = d.t[1];
          for (int t = 0; t < n; ++t) {
            const int first = alt ? t & 1 : 0, last = alt ? first : (d.n[1] > 0 ? 1 : 0), step = alt ? 2 : 1;
#pragma unroll 1
            for (int b = first; b <= last; ++b) is.pv(b, t < step, t + step >= n);
            is.free_v();
          }
        }
        commit<C>(&mi.mma_done);
      }
      __syncwarp();
    }
  } else if (warp >= WARP_EPI) {
    // ================================================================ epilogue: thread = query row
    setmaxnreg_dec<REGS_PARALLEL.epilogue>();
    const int r = tid & 127, wi = r % w;
    const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const bool sectors = (reinterpret_cast<uintptr_t>(prm.part_o) & 31) == 0;  // a workspace is aligned to 16 bytes only
    uint32_t nd = 0, nq = 0, no[2] = {0, 0};
    while (true) {
      const Desc d = next_desc<C>(cx, nd, true);
      if (d.kind == KIND_DONE) break;
#pragma unroll 1
      for (int b0 = 0; b0 < (alt ? 1 : 2); ++b0) {
        // one output block: block b0, or with alt the sum of both (the second may have had no tile)
        if ((b0 ? d.n[1] : d.n[0]) == 0) continue;
        const bool two = alt && d.n[1] > 0;
        float m = -INFINITY, f[2] = {0.0f, 0.0f}, l = 0.0f;
        {
          float mb[2] = {-INFINITY, -INFINITY}, lb[2] = {0.0f, 0.0f};
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int b = alt ? i : b0;
            if (i == 1 && !two) break;
            const uint32_t ph = b ? no[1] : no[0];
            WAIT2(&mi.lm_full[b], full_par(ph), W2_LM);
            mb[i] = mi.lm[b][0][r];
            lb[i] = mi.lm[b][1][r];
            warp_arrive(&mi.lm_free[b]);
            WAIT2S(&mi.o_full[b], full_par(ph), W2_OFULL);
            if (b) ++no[1]; else ++no[0];
          }
          m = fmaxf(mb[0], mb[1]);
#pragma unroll
          for (int i = 0; i < 2; ++i) f[i] = mb[i] == -INFINITY ? 0.0f : fast_exp2(mb[i] - m);
          l = f[0] * lb[0] + f[1] * lb[1];
        }
        tc_fence_after_sync();
        if (r == 0) mbar_arrive(&mi.q_free[nq % NQ]);                        // every MMA that reads the query slot has completed
        ++nq;
        const int g = first_head(d.h[0], b0, rank) + r / w;
        const bool valid = g < G;
        const int h = d.hkv * G + g;
        const bool whole = prm.n_split == 1;
        if (whole) { const float inv = 1.0f / l; f[0] *= inv; f[1] *= inv; }
        const size_t prow = (((size_t)d.c * prm.Hq + h) * prm.n_split + d.len) * w + wi;
        uint4* const out = whole ? reinterpret_cast<uint4*>(prm.out + (((size_t)d.c * w + wi) * prm.Hq + h) * D)
                                 : reinterpret_cast<uint4*>(prm.part_o + prow * D);
        const uint32_t tO = cx.tmem + C::TM_O + (alt ? 0 : b0 * D) + lane_sel;
#pragma unroll 1
        for (int q = 0; q < D / 16; ++q) {
          uint32_t oa[16], ob[16];
          tmem_ld16(tO + q * 16, oa);
          if (two) tmem_ld16(tO + D + q * 16, ob);
          tmem_wait_ld();
          float x[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            asm volatile("" : "+r"(oa[i]));                                  // no use moves above the wait
            x[i] = __uint_as_float(oa[i]) * f[0];
          }
          if (two) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              asm volatile("" : "+r"(ob[i]));
              x[i] = fmaf(__uint_as_float(ob[i]), f[1], x[i]);
            }
          }
          if (valid && whole) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
              out[q * 2 + i] = make_uint4(pack_bf16x2(x[i * 8], x[i * 8 + 1]), pack_bf16x2(x[i * 8 + 2], x[i * 8 + 3]),
                                          pack_bf16x2(x[i * 8 + 4], x[i * 8 + 5]), pack_bf16x2(x[i * 8 + 6], x[i * 8 + 7]));
          } else if (valid) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (!sectors) out[q * 4 + i] = make_uint4(__float_as_uint(x[i * 4]), __float_as_uint(x[i * 4 + 1]), __float_as_uint(x[i * 4 + 2]),
                                                        __float_as_uint(x[i * 4 + 3]));
              else if (i % 2 == 0) st_global_f32x8(out + q * 4 + i, &x[i * 4]);
          }
        }
        warp_arrive_leader(in_cta<C>(&mi.o_free[alt ? 0 : b0], 0));
        if (two) warp_arrive_leader(in_cta<C>(&mi.o_free[1], 0));
        if (valid && !whole) reinterpret_cast<float2*>(prm.part_ml)[prow] = make_float2(m, l);
        if (valid && whole && prm.lse_out)
          prm.lse_out[((size_t)d.c * prm.Hq + h) * w + wi] = (m + log2f(l)) * 0.6931471805599453f;
      }
    }
  } else {
    // ================================================================ softmax
    setmaxnreg_inc<REGS_PARALLEL.softmax>();
    const int b = warp >> 2;
    const int r = tid & 127, wi = r % w;
    const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tS = cx.tmem + C::tm_s(b) + lane_sel, tP = cx.tmem + C::TM_P + b * 64 + lane_sel;
    const uint32_t tO = cx.tmem + C::TM_O + b * D + lane_sel;
    const float scale_log2 = prm.scale_log2;
    Hooks<C> hk(cx, b);
    uint32_t nd = 0, n_s = 0, n_blk = 0;
    while (true) {
      const Desc d = next_desc<C>(cx, nd, true);
      if (d.kind == KIND_DONE) break;
      const int n = b ? d.n[1] : d.n[0];
      if (n == 0) continue;
      RowState st = {-INFINITY, 0.0f};
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        const int j = d.t[0] + (alt ? 2 * i + b : i);
        const int vis = j == prm.n_cache_tiles ? wi + 1 : prm.Nk - j * TILE;     // window tile: causal; ragged last cache tile
        WAIT2S(&mi.s_full[b], full_par(n_s), W2_SFULL);
        ++n_s;
        tc_fence_after_sync();
        if (i > 0 && j != prm.n_cache_tiles && vis >= TILE) softmax_tile<D, false>(tS, tP, tO, TILE, false, scale_log2, st, hk);
        else softmax_tile<D, true>(tS, tP, tO, vis, i == 0, scale_log2, st, hk);
        ++hk.tiles;
      }
      WAIT2S(&mi.lm_free[b], free_par(n_blk), W2_LMFREE);
      ++n_blk;
      mi.lm[b][0][r] = st.m;
      mi.lm[b][1][r] = st.l;
      warp_arrive(&mi.lm_full[b]);
    }
  }

  teardown<C>(cx);
}

// Merge of the key splits: out = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s.  One warp per output row, a lane per
// split for the weights; the rows' loads are independent of one another.
template <int D>
__global__ void __launch_bounds__(128) parallel_merge_kernel(const float* __restrict__ part_o, const float* __restrict__ part_ml,
                                                             int n_rows, int w, int Hq, int n_split,
                                                             __nv_bfloat16* __restrict__ out, float* __restrict__ lse_out) {
  chain();
  const int row = blockIdx.x * 4 + (threadIdx.x >> 5);                       // (seq * Hq + h) * w + i
  const int lane = threadIdx.x & 31;
  if (row >= n_rows) return;
  const int bh = row / w, i = row % w;
  const float2* const ml = reinterpret_cast<const float2*>(part_ml) + (size_t)bh * n_split * w + i;
  float m = -INFINITY;
  for (int s = lane; s < n_split; s += 32) m = fmaxf(m, ml[(size_t)s * w].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  float denom = 0.0f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  const float* const po = part_o + ((size_t)bh * n_split * w + i) * D;
  for (int s0 = 0; s0 < n_split; s0 += 32) {
    const float2 mine = s0 + lane < n_split ? ml[(size_t)(s0 + lane) * w] : make_float2(-INFINITY, 0.0f);
    const float wgt = exp2f(mine.x - m);
    denom += wgt * mine.y;
    const int ns = n_split - s0 < 32 ? n_split - s0 : 32;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) {
      const float ws = __shfl_sync(0xFFFFFFFFu, wgt, s);
      if (lane < D / 4) {
        const float4 o = __ldg(reinterpret_cast<const float4*>(po + (size_t)(s0 + s) * w * D) + lane);
        acc.x += ws * o.x; acc.y += ws * o.y; acc.z += ws * o.z; acc.w += ws * o.w;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) denom += __shfl_xor_sync(0xFFFFFFFFu, denom, o);
  const float inv = 1.0f / denom;
  const int seq = bh / Hq, h = bh % Hq;
  if (lane < D / 4)
    reinterpret_cast<uint2*>(out + (((size_t)seq * w + i) * Hq + h) * D)[lane] =
        make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
  if (lane == 0 && lse_out) lse_out[row] = (m + log2f(denom)) * 0.6931471805599453f;
}

// ====================================================================================
//                                   host launcher
// ====================================================================================
template <int D, bool PAIR>
static cudaError_t launch_parallel_t(const CUtensorMap* maps, const ParallelParams& prm, int sm_count, cudaStream_t st) {
  using C = Cfg<D, PAIR>;
  // the opt-in to large dynamic shared memory is a per-device attribute of the function: set it on every call
  // (a host-side call of a few hundred nanoseconds) rather than remember which devices have it
  if (cudaError_t e = cudaFuncSetAttribute(parallel_attn_kernel<D, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, Off<C>::TOTAL);
      e != cudaSuccess) return e;
  const long long n_items = (long long)prm.B * prm.Hkv * prm.n_rg * prm.n_split;
  const int units = sm_count / C::NCTA;
  if (units < 1) return cudaErrorInvalidConfiguration;
  if (cudaError_t e = launch_chained(parallel_attn_kernel<D, PAIR>, dim3((unsigned)((n_items < units ? (int)n_items : units) * C::NCTA)), dim3(NT2),
                                     Off<C>::TOTAL, st, C::NCTA, maps[0], maps[1], maps[2], maps[3], maps[4], prm);
      e != cudaSuccess) return e;
  if (prm.n_split > 1) {
    const int rows = prm.B * prm.Hq * prm.w;
    return launch_chained(parallel_merge_kernel<D>, dim3((rows + 3) / 4), dim3(128), 0, st, 1, prm.part_o, prm.part_ml, rows, prm.w, prm.Hq,
                          prm.n_split, prm.out, prm.lse_out);
  }
  return cudaSuccess;
}

cudaError_t launch_parallel_attn(const CUtensorMap* maps, const ParallelParams& prm, int d, bool pair, int sm_count, cudaStream_t st) {
  if (d == 64) return launch_parallel_t<64, false>(maps, prm, sm_count, st);
  return pair ? launch_parallel_t<128, true>(maps, prm, sm_count, st) : launch_parallel_t<128, false>(maps, prm, sm_count, st);
}

}  // namespace pc
