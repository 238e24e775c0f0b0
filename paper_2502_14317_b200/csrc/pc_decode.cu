// Parallel (global) attention for few query rows (Eq. 9-11): decoding steps and short query windows, up to 32 rows
// (q-heads of a kv-head x window tokens) per (sequence, kv-head).  One launch: rotation of the queries, attention
// over the cache and the window's own keys, merge of the key splits, append of the new entries.
//
// Bound by reading the cache once, so everything else has to stay small beside 64 KB of K and V per 128 keys.  With the
// query rows as the M = 128 rows of an MMA (the kernel for wide windows) a decoding step of 4 rows computes 32 times
// the products and exponentials that it needs, and the board power cap then slows the memory down as well.  Here the
// products are transposed: keys (then head-dim columns) are the M = 128 rows, the query rows are the N = 16 or 32
// columns:
//     S^T [128 keys x N] = K_tile Q^T        thread = key, a register per query row
//     O^T [d x N]       += V_tile^T P^T      P^T goes through shared memory, N x 128 keys
// The reference maximum of a row is shared by all keys through shared memory; a tile whose logits stay below
// 2^8 times it needs one barrier vote and no reduction over keys.  Row sums stay per thread until the end.
//
// A (sequence, kv-head) is split over the CTAs of a cluster (1 to 16), which merge through distributed shared memory.
// Many items: two CTAs per SM, three 32 KB stages each, the prologue of one under the copies of the other.  Few items of head size
// 128, where a CTA alone must take its tiles fast: one CTA per SM with six stages (rule and figures: few_plan in pc_api.cu).
//
// What bounds it: many sequences, the copy bandwidth; one sequence, latencies - of 39 K cycles over 16401 entries (one token,
// 8 kv-heads, ten CTAs each, caches cold) 27 K pass in the tiles, 3 K before the queries are asked for (their
// angles, under the kernel ahead where there is one), 5 K in the queries' rotation, 4 K in the merge.
//
// Measured on caches of 16401 entries, 32 q-heads over 8 kv-heads of size 128, against the row-major kernel with its
// five other launches: 64 sequences, one token 867 -> 642 us (6.7 TB/s, the copy bandwidth); one sequence 46.6 -> 16.7 us
// (28.7 with three stages everywhere, a load per query row where it is used and the splits read one after the other
// in the merge).  8 tokens, 4096 entries, one sequence: 20.4 -> 13.2 us with those three changed.
// 32 rows (64 sequences, 8 tokens, 8000 entries): 521 -> 434 us.  With 64 rows the chain of a tile (64 exponentials a
// thread between two products) outlasts the copies: 500 -> 626 us, so those stay with the row-major kernel.
// Warps: 0-3 softmax and epilogue, 4 TMA producer, 5 MMA issuer; all but 4 rotate queries first.
#include "pc_attn.h"
#include "pc_kernels.h"
#include "pc_softmax.cuh"
#include <cfloat>

namespace pc {

namespace {

constexpr int TILE = 128;
constexpr int NTD = 256;
constexpr int WARP_PRODUCER = 4, WARP_MMA = 5;
constexpr int MAX_STAGES = 6;

enum { WD_KV = 301, WD_FREE, WD_S, WD_P, WD_PV };

// DEEP: twice the stages, one CTA per SM (head size 128 only)
template <int D, int N, bool DEEP>
struct Lay {
  static constexpr int TILE_BYTES = TILE * D * 2;
  static constexpr int NS = (D == 128 ? 3 : 6) * (DEEP ? 2 : 1);
  static constexpr int OFF_Q = NS * TILE_BYTES;
  static constexpr int OFF_P = OFF_Q + N * D * 2;
  static constexpr int OFF_MISC = OFF_P + N * TILE * 2;
  static constexpr int TMEM_COLS = N == 16 ? 64 : 128;      // two S^T buffers and O^T
};
template <int N>
struct __align__(16) Misc {
  uint64_t kv_full[MAX_STAGES], kv_free[MAX_STAGES];
  uint64_t s_full[2], p_full, pv_done, mma_done;
  uint32_t tmem_base;
  int abort_flag;                  // these two words stay adjacent: bounded waits read the limit through the flag's address
  int wait_kcycles;
  alignas(16) float negm[N];       // minus the reference maximum of a row (log2 units)
  alignas(16) float red[4][N];                 // per warp: row maxima, then row sums
};

__device__ __forceinline__ uint32_t full_par(uint32_t n) { return n & 1u; }
__device__ __forceinline__ uint32_t free_par(uint32_t n) { return (n & 1u) ^ 1u; }
__device__ __forceinline__ bool any_of_128(bool x) {               // OR over the four softmax warps
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"(static_cast<uint32_t>(x)) : "memory");
  return r != 0;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float warp_max(float x) {               // order-preserving map to int, one redux
  int i = __float_as_int(x);
  i ^= (i >> 31) & 0x7FFFFFFF;
  i = __reduce_max_sync(0xFFFFFFFFu, i);
  return __int_as_float(i ^ ((i >> 31) & 0x7FFFFFFF));
}
// Sums over the lanes of N values per lane: the sum of x[i] in lane i (N = 16: also in lane i + 16).  Halves the values a lane
// holds with every exchange, N - 1 exchanges in all instead of 5 N.
template <int N>
__device__ __forceinline__ float lane_sums(float (&x)[N], int lane) {
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const float give = upper ? x[j] : x[j + o], keep = upper ? x[j + o] : x[j];
      x[j] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
    }
  }
  return N == 16 ? x[0] + __shfl_xor_sync(0xFFFFFFFFu, x[0], 16) : x[0];
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
// sum over the CTAs s < ns of weight[s] * (four floats at addr in CTA s); all reads are in flight together
template <int MAX>
__device__ __forceinline__ float4 sum_splits(const float* addr, const float* weight, int ns, int self) {
  float4 x[MAX], acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
  for (int s = 0; s < MAX; ++s) x[s] = ld_cluster_f32x4(map_to_cta(addr, s < ns ? s : self));   // (weight 0 there)
#pragma unroll
  for (int s = 0; s < MAX; ++s) {
    acc.x = fmaf(weight[s], x[s].x, acc.x); acc.y = fmaf(weight[s], x[s].y, acc.y);
    acc.z = fmaf(weight[s], x[s].z, acc.z); acc.w = fmaf(weight[s], x[s].w, acc.w);
  }
  return acc;
}
template <int N>
__device__ __forceinline__ void load_cols(uint32_t taddr, float (&s)[N]) {
  uint32_t a[N];
  if constexpr (N == 16) tmem_ld16(taddr, a); else tmem_ld32(taddr, a);
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < N; ++i) { asm volatile("" : "+r"(a[i])); s[i] = __uint_as_float(a[i]); }   // no use moves above the wait
}

}  // namespace

template <int D, int N, bool DEEP>
__global__ void __launch_bounds__(NTD, DEEP ? 1 : 2)
decode_attn_kernel(const __grid_constant__ CUtensorMap tm_kc, const __grid_constant__ CUtensorMap tm_vc,
                   const __grid_constant__ CUtensorMap tm_kw, const __grid_constant__ CUtensorMap tm_vw,
                   const __grid_constant__ DecodeParams prm) {
  using Y = Lay<D, N, DEEP>;
  // Pause between two polls: none where a CTA has its SM for itself (few items, every wait on the chain of a tile): one token over a
  // cache of 16401 15.60 -> 15.38 us, over two of 16000 25.27 -> 25.15, 2 over eight of 4000, 28/4 heads 15.98 -> 15.88.  With two CTAs an
  // SM it helps some shapes and costs others: 4 over eight of 9000, head size 64 35.8 -> 34.6, 2 over 32 of 16000 159 -> 161.
  constexpr unsigned POLL_NS = DEEP ? 0 : SPIN_BACKOFF_NS;
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc<N>& mi = *reinterpret_cast<Misc<N>*>(smem + Y::OFF_MISC);
  volatile int* const abort_flag = &mi.abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ns = prm.n_split, split = blockIdx.x % ns, item = blockIdx.x / ns;      // the CTAs of a cluster are one item's splits
  const int hkv = item % prm.Hkv, seq = item / prm.Hkv;
  const int G = prm.Hq / prm.Hkv, w = prm.w, R = G * w;
  const int n_all = prm.n_cache_tiles + 1;                                          // the last tile holds the window's own keys
  const int j0 = (int)((long long)n_all * split / ns), j1 = (int)((long long)n_all * (split + 1) / ns), n = j1 - j0;
  const uint32_t sK = smem_u32(smem), sQ = sK + Y::OFF_Q, sP = sK + Y::OFF_P;

  // copies of tile i of this split into the next two stages (K, then V)
  auto load_half = [&](uint32_t kv) {
    const int st = kv % Y::NS, j = j0 + (int)(kv >> 1);
    uint8_t* const dst = smem + st * Y::TILE_BYTES;
    mbar_arrive_expect_tx(&mi.kv_full[st], Y::TILE_BYTES);
    for (int a = 0; a < D / 64; ++a) {
      if (j < prm.n_cache_tiles) tma_load_4d(dst + a * 16384, (kv & 1) ? &tm_vc : &tm_kc, &mi.kv_full[st], a * 64, j * TILE, hkv, seq);
      else tma_load_4d(dst + a * 16384, (kv & 1) ? &tm_vw : &tm_kw, &mi.kv_full[st], a * 64, hkv, 0, seq);
    }
  };
  const uint32_t n_kv = 2 * (uint32_t)n, n_first = n_kv < (uint32_t)Y::NS ? n_kv : (uint32_t)Y::NS;

  if (warp == WARP_PRODUCER) {
    if (elect_one()) {
      for (int i = 0; i < Y::NS; ++i) { mbar_init(&mi.kv_full[i], 1); mbar_init(&mi.kv_free[i], 1); }
      mbar_init(&mi.s_full[0], 1); mbar_init(&mi.s_full[1], 1);
      mbar_init(&mi.p_full, 4); mbar_init(&mi.pv_done, 1); mbar_init(&mi.mma_done, 1);
      mi.abort_flag = 0;
      mi.wait_kcycles = prm.wait_kcycles;
      fence_mbar_init();
      chain();
      for (uint32_t kv = 0; kv < n_first; ++kv) load_half(kv);
    }
    __syncwarp();
  } else {
    if (warp == WARP_MMA) tmem_alloc(&mi.tmem_base, Y::TMEM_COLS);
    // ---- rotate the queries: the fp64 rotation rounded once to bf16, row g * w + i of the operand
    constexpr int HALF = D / 2;
    const int rt = warp > WARP_PRODUCER ? tid - 32 : tid;                           // 0 .. 223
    const uint16_t* const qs = reinterpret_cast<const uint16_t*>(prm.q_win) + ((size_t)seq * w * prm.Hq + (size_t)hkv * G) * D;
    auto q_slot = [&](int r, int e) -> uint16_t* {
      return reinterpret_cast<uint16_t*>(smem + Y::OFF_Q + (e / 64) * (N * 128) + sw128_offset(r, (e % 64) / 8) + (e % 8) * 2);
    };
    // a thread keeps its pair over the tokens: one pow, and the angles of its first tokens need nothing from before this launch
    constexpr int TURNERS = (NTD - 32) / HALF * HALF, STEP = TURNERS / HALF, AHEAD = 3;
    const int t = rt % HALF, i_first = rt < TURNERS ? rt / HALF : w;
    double sn[AHEAD], cs[AHEAD], freq = 0.0;
    auto turn = [&](int i, double& s, double& c) { sincos((double)(prm.q_pos0 + i) * freq, &s, &c); };
    if (i_first < w) freq = pow((double)prm.rope_theta, -2.0 * (double)t / (double)D);
#pragma unroll
    for (int k = 0; k < AHEAD; ++k)
      if (i_first + k * STEP < w) turn(i_first + k * STEP, sn[k], cs[k]);
    chain();
    // the rows as they are first go to the P buffer, all loads in flight at once (a load per row and pair where it is needed
    // puts their latencies in a row)
    uint16_t* const raw = reinterpret_cast<uint16_t*>(smem + Y::OFF_P);             // [token * G + g][D]
    for (int e = rt; e < R * (D / 8); e += NTD - 32) {
      const int i = e / (G * (D / 8)), c = e - i * (G * (D / 8));
      reinterpret_cast<uint4*>(raw)[e] = __ldg(reinterpret_cast<const uint4*>(qs + (size_t)i * prm.Hq * D) + c);
    }
    named_barrier_sync(3, NTD - 32);
    auto rotate = [&](int i, double s, double c) {
#pragma unroll 4
      for (int g = 0; g < G; ++g) {
        const uint16_t* const x = raw + (i * G + g) * D + t;
        const double a = (double)__uint_as_float((uint32_t)x[0] << 16), b = (double)__uint_as_float((uint32_t)x[HALF] << 16);
        *q_slot(g * w + i, t) = f64_to_bf16_rne(a * c - b * s);
        *q_slot(g * w + i, t + HALF) = f64_to_bf16_rne(b * c + a * s);
      }
    };
#pragma unroll
    for (int k = 0; k < AHEAD; ++k)
      if (i_first + k * STEP < w) rotate(i_first + k * STEP, sn[k], cs[k]);
    for (int i = i_first + AHEAD * STEP; i < w; i += STEP) {
      double s, c;
      turn(i, s, c);
      rotate(i, s, c);
    }
    // operand rows that are no query rows: zero queries and zero probabilities
    for (int e = rt; e < (N - R) * (D / 8); e += NTD - 32) {
      const int r = R + e / (D / 8), c = e % (D / 8);
      *reinterpret_cast<uint4*>(smem + Y::OFF_Q + (c / 8) * (N * 128) + sw128_offset(r, c % 8)) = make_uint4(0, 0, 0, 0);
    }
    named_barrier_sync(3, NTD - 32);
    for (int e = rt; e < (N - R) * (TILE / 8); e += NTD - 32) {
      const int r = R + e / (TILE / 8), c = e % (TILE / 8);
      *reinterpret_cast<uint4*>(smem + Y::OFF_P + (c / 8) * (N * 128) + sw128_offset(r, c % 8)) = make_uint4(0, 0, 0, 0);
    }
    if (rt < N) mi.negm[rt] = INFINITY;
    // ---- append: the attention never reads entries from Nk on, so the new ones can be written at any time
    if (prm.k_append != nullptr && split == 0) {
      const uint4* const kw = reinterpret_cast<const uint4*>(prm.k_win);
      const uint4* const vw = reinterpret_cast<const uint4*>(prm.v_win);
      uint4* const kd = reinterpret_cast<uint4*>(prm.k_append);
      uint4* const vd = reinterpret_cast<uint4*>(prm.v_append);
      for (int e = rt; e < w * (D / 8); e += NTD - 32) {
        const int i = e / (D / 8), c = e % (D / 8);
        const size_t src = (((size_t)seq * w + i) * prm.Hkv + hkv) * (D / 8) + c;
        const size_t dst = (((size_t)seq * prm.Hkv + hkv) * prm.Nk_cap + prm.Nk + i) * (D / 8) + c;
        kd[dst] = __ldg(kw + src);
        vd[dst] = __ldg(vw + src);
      }
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();
  }
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = mi.tmem_base, tO = tmem + 2 * N;

  if (warp == WARP_PRODUCER) {
    if (elect_one()) {
      uint32_t kv = n_first;
      for (; kv < n_kv && !*abort_flag; ++kv) {
        if (!mbar_wait_ns<POLL_NS>(&mi.kv_free[kv % Y::NS], free_par(kv / Y::NS), abort_flag, prm.status, WD_FREE)) break;
        load_half(kv);
      }
      for (uint32_t i = kv > (uint32_t)Y::NS ? kv - Y::NS : 0; i < kv; ++i)             // every copy has landed before exit
        mbar_wait_drain(&mi.kv_full[i % Y::NS], full_par(i / Y::NS), abort_flag);
    }
    __syncwarp();
  } else if (warp == WARP_MMA) {
    if (elect_one()) {
      constexpr uint32_t idesc_qk = make_idesc_bf16_f32(128, N, false, false), idesc_pv = make_idesc_bf16_f32(128, N, true, false);
      // S^T of tile i into buffer i & 1; head size 64: the second half of the 128 accumulator rows repeats rows of the
      // first (its operand starts 8 keys further in the same stage) and is never read
      constexpr uint32_t V_LBO = D == 128 ? 16384 : 1024;
      auto issue_qk = [&](int i) {
        const uint32_t kv = 2 * (uint32_t)i, st = kv % Y::NS;
        mbar_wait_ns<POLL_NS>(&mi.kv_full[st], full_par(kv / Y::NS), abort_flag, prm.status, WD_KV);
        tc_fence_after_sync();
        const uint32_t k = sK + st * Y::TILE_BYTES;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          mma_ss(tmem + (i & 1) * N, make_smem_desc_sw128(k + (ks / 4) * 16384 + (ks % 4) * 32, 16, 1024),
                 make_smem_desc_sw128(sQ + (ks / 4) * (N * 128) + (ks % 4) * 32, 16, 1024), idesc_qk, ks > 0);
        mma_commit(&mi.s_full[i & 1]);
        mma_commit(&mi.kv_free[st]);
      };
      issue_qk(0);
      for (int i = 0; i < n && !*abort_flag; ++i) {
        if (i + 1 < n) issue_qk(i + 1);                       // P of tile i-1 was there, so its S buffer has been read
        const uint32_t kv = 2 * (uint32_t)i + 1, st = kv % Y::NS;
        mbar_wait_ns<POLL_NS>(&mi.kv_full[st], full_par(kv / Y::NS), abort_flag, prm.status, WD_KV);
        mbar_wait_ns<POLL_NS>(&mi.p_full, full_par(i), abort_flag, prm.status, WD_P);
        tc_fence_after_sync();
        const uint32_t v = sK + st * Y::TILE_BYTES;
#pragma unroll
        for (int ks = 0; ks < TILE / 16; ++ks)
          mma_ss(tO, make_smem_desc_sw128(v + ks * 2048, V_LBO, 1024),
                 make_smem_desc_sw128(sP + (ks / 4) * (N * 128) + (ks % 4) * 32, 16, 1024), idesc_pv, i > 0 || ks > 0);
        mma_commit(&mi.kv_free[st]);
        mma_commit(&mi.pv_done);
      }
      mma_commit(&mi.mma_done);
    }
    __syncwarp();
  } else if (warp < 4) {
    // ================================================================ softmax: thread = key of the tile
    const uint32_t lane_sel = static_cast<uint32_t>(warp * 32) << 16;
    const float scale = prm.scale_log2;
    float l[N];
#pragma unroll
    for (int r = 0; r < N; ++r) l[r] = 0.0f;
    for (int i = 0; i < n; ++i) {
      mbar_wait_ns<POLL_NS>(&mi.s_full[i & 1], full_par(i >> 1), abort_flag, prm.status, WD_S);
      tc_fence_after_sync();
      float s[N];
      load_cols<N>(tmem + (i & 1) * N + lane_sel, s);
      const int j = j0 + i;
      if (j == prm.n_cache_tiles) {                           // the window's own keys: causal
        int wi = 0;
#pragma unroll
        for (int r = 0; r < N; ++r) {
          if (tid > wi) s[r] = -INFINITY;
          if (++wi == w) wi = 0;
        }
      } else if (j * TILE + tid >= prm.Nk) {                  // ragged last cache tile
#pragma unroll
        for (int r = 0; r < N; ++r) s[r] = -INFINITY;
      }
      bool raise = i == 0;
#pragma unroll
      for (int q = 0; q < N / 8; ++q) {                       // rows in groups of 8 (those that are no query rows come out finite)
        if (q * 8 < R) {
          const float4 na = reinterpret_cast<const float4*>(mi.negm)[2 * q], nb = reinterpret_cast<const float4*>(mi.negm)[2 * q + 1];
          const float nm[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
          float x = fmaf(s[q * 8], scale, nm[0]);
#pragma unroll
          for (int r = 1; r < 8; ++r) x = fmaxf(x, fmaf(s[q * 8 + r], scale, nm[r]));
          raise |= x > LAZY_RESCALE_LOG2;
        }
      }
      if (any_of_128(raise)) {                                // rare after the first tile: raise the reference maxima
#pragma unroll
        for (int r = 0; r < N; ++r) {
          const float m = warp_max(s[r]);
          if (lane == 0) mi.red[warp][r] = m * scale;
        }
        named_barrier_sync(1, 128);
        float m_old = 0.0f, m_new = 0.0f;
        if (tid < N) {
          m_old = -mi.negm[tid];
          m_new = fmaxf(fmaxf(fmaxf(mi.red[0][tid], mi.red[1][tid]), fmaxf(mi.red[2][tid], mi.red[3][tid])), m_old);
          m_new = fmaxf(m_new, -FLT_MAX);                     // every logit so far -inf: the probabilities are 0, not exp2(-inf + inf)
        }
        named_barrier_sync(1, 128);
        if (tid < N) {
          mi.negm[tid] = -m_new;
          mi.red[0][tid] = m_old == -INFINITY ? 0.0f : fast_exp2(m_old - m_new);
        }
        named_barrier_sync(1, 128);
        if (i > 0) {
          mbar_wait_ns<POLL_NS>(&mi.pv_done, full_par(i - 1), abort_flag, prm.status, WD_PV);
          tc_fence_after_sync();
          float o[N];
          load_cols<N>(tO + lane_sel, o);
#pragma unroll
          for (int q = 0; q < N / 8; ++q) {
            uint32_t a[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) a[r] = __float_as_uint(o[q * 8 + r] * mi.red[0][q * 8 + r]);
            tmem_st8(tO + lane_sel + q * 8, a);
          }
          tmem_wait_st();
        }
#pragma unroll
        for (int r = 0; r < N; ++r) l[r] *= mi.red[0][r];
      }
      if (i > 0) mbar_wait_ns<POLL_NS>(&mi.pv_done, full_par(i - 1), abort_flag, prm.status, WD_PV);   // P of the tile before has been read
      uint8_t* const pdst = smem + Y::OFF_P + (tid / 64) * (N * 128) + (tid % 8) * 2;
#pragma unroll
      for (int q = 0; q < N / 8; ++q) {
        if (q * 8 < R) {
          const float4 na = reinterpret_cast<const float4*>(mi.negm)[2 * q], nb = reinterpret_cast<const float4*>(mi.negm)[2 * q + 1];
          const float nm[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
          float pr[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) { pr[r] = fast_exp2(fmaf(s[q * 8 + r], scale, nm[r])); l[q * 8 + r] += pr[r]; }
#pragma unroll
          for (int r = 0; r < 8; ++r)
            *reinterpret_cast<__nv_bfloat16*>(pdst + sw128_offset(q * 8 + r, (tid % 64) / 8)) = __float2bfloat16_rn(pr[r]);
        }
      }
      fence_proxy_async_smem();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&mi.p_full);
    }
    // ---- row sums over the keys, then O^T (thread = head-dim column)
    mbar_wait_ns<POLL_NS>(&mi.pv_done, full_par(n - 1), abort_flag, prm.status, WD_PV);
    tc_fence_after_sync();
    const float row_sum = lane_sums<N>(l, lane);
    if (lane < N) mi.red[warp][lane] = row_sum;
    named_barrier_sync(1, 128);
    float o[N];
    load_cols<N>(tO + lane_sel, o);
    if (ns == 1) {
      __nv_bfloat16* const out = prm.out + ((size_t)seq * w * prm.Hq + (size_t)hkv * G) * D + tid;
      int g = 0, wi = 0;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (r < R && tid < D) {
          const float lt = (mi.red[0][r] + mi.red[1][r]) + (mi.red[2][r] + mi.red[3][r]);
          out[((size_t)wi * prm.Hq + g) * D] = __float2bfloat16_rn(o[r] / lt);
        }
        if (++wi == w) { wi = 0; ++g; }
      }
      if (prm.lse_out != nullptr && tid < R) {
        const float lt = (mi.red[0][tid] + mi.red[1][tid]) + (mi.red[2][tid] + mi.red[3][tid]);
        prm.lse_out[((size_t)seq * prm.Hq + hkv * G) * w + tid] = (log2f(lt) - mi.negm[tid]) * 0.6931471805599453f;
      }
    } else {
      float* const part = reinterpret_cast<float*>(smem);     // [row][d]; the ring is idle: everything has been consumed
#pragma unroll
      for (int r = 0; r < N; ++r)
        if (r < R && tid < D) part[r * D + tid] = o[r];
    }
  }

  if (ns > 1) {
    // ---- merge of the splits: every CTA takes a slice of the output.  First the weights of the splits in its rows, a warp
    // per row and a lane per split, then the sums; the remote reads of a step are all in flight together.
    cluster_sync_all();
    const int total = R * D, chunk = (total / 4 + ns - 1) / ns * 4, e0 = split * chunk, e1 = e0 + chunk < total ? e0 + chunk : total;
    float* const weight = reinterpret_cast<float*>(smem + Y::TILE_BYTES);           // [row][16], behind the partial results
    for (int r = e0 / D + warp; r * D < e1; r += NTD / 32) {
      float m = -INFINITY, l = 0.0f;
      if (lane < ns) {
        m = -ld_cluster_f32(map_to_cta(&mi.negm[r], lane));
        l = (ld_cluster_f32(map_to_cta(&mi.red[0][r], lane)) + ld_cluster_f32(map_to_cta(&mi.red[1][r], lane))) +
            (ld_cluster_f32(map_to_cta(&mi.red[2][r], lane)) + ld_cluster_f32(map_to_cta(&mi.red[3][r], lane)));
      }
      float top = m;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
      const float f = lane < ns ? exp2f(m - top) : 0.0f;
      float sum = f * l;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
      if (lane < 16) weight[r * 16 + lane] = f / sum;
      if (prm.lse_out != nullptr && lane == 0 && r * D >= e0)
        prm.lse_out[((size_t)seq * prm.Hq + hkv * G) * w + r] = (top + log2f(sum)) * 0.6931471805599453f;
    }
    __syncthreads();
    for (int e = e0 + 4 * tid; e < e1; e += 4 * NTD) {
      const int r = e / D, dd = e % D, wi = r % w, g = r / w;
      const float* const part = reinterpret_cast<const float*>(smem) + e;
      const float* const wr = weight + r * 16;
      const float4 o = ns > 8 ? sum_splits<16>(part, wr, ns, split) : ns > 4 ? sum_splits<8>(part, wr, ns, split) :
                       ns > 2 ? sum_splits<4>(part, wr, ns, split) : sum_splits<2>(part, wr, ns, split);
      *reinterpret_cast<uint2*>(prm.out + (((size_t)seq * w + wi) * prm.Hq + hkv * G + g) * D + dd) =
          make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
    }
    cluster_sync_all();                                       // no CTA exits while another may read its shared memory
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == WARP_MMA) {
    mbar_wait_drain(&mi.mma_done, 0, abort_flag);             // immediate in a clean run; after an abort no MMA may still run
    tc_fence_after_sync();
    tmem_dealloc(tmem, Y::TMEM_COLS);
  }
}

template <int D, int N, bool DEEP>
static cudaError_t prepare(int n_split) {
  using Y = Lay<D, N, DEEP>;
  constexpr int SMEM = Y::OFF_MISC + (int)sizeof(Misc<N>);
  static_assert((DEEP ? 1 : 2) * (SMEM + 1024) <= 233472, "CTAs per SM");
  auto* const kernel = decode_attn_kernel<D, N, DEEP>;
  if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM); e != cudaSuccess) return e;
  return n_split > 8 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess;
}
template <int D, int N, bool DEEP>
static cudaError_t launch_decode_t(const CUtensorMap* maps, const DecodeParams& prm, cudaStream_t st) {
  if (cudaError_t e = prepare<D, N, DEEP>(prm.n_split); e != cudaSuccess) return e;
  return launch_chained(decode_attn_kernel<D, N, DEEP>, dim3((unsigned)(prm.B * prm.Hkv * prm.n_split)), dim3(NTD),
                        Lay<D, N, DEEP>::OFF_MISC + sizeof(Misc<N>), st, prm.n_split, maps[0], maps[1], maps[2], maps[3], prm);
}
template <int D, int N>
static cudaError_t launch_decode_n(const CUtensorMap* maps, const DecodeParams& prm, cudaStream_t st) {
  if constexpr (D == 128)
    if (prm.deep) return launch_decode_t<D, N, true>(maps, prm, st);
  return launch_decode_t<D, N, false>(maps, prm, st);
}

cudaError_t launch_decode_attn(const CUtensorMap* maps, const DecodeParams& prm, int d, cudaStream_t st) {
  const int rows = prm.Hq / prm.Hkv * prm.w;
  if (d == 128) return rows <= 16 ? launch_decode_n<128, 16>(maps, prm, st) : launch_decode_n<128, 32>(maps, prm, st);
  return rows <= 16 ? launch_decode_n<64, 16>(maps, prm, st) : launch_decode_n<64, 32>(maps, prm, st);
}

template <bool DEEP>
static int clusters_t(int n_split) {                          // the largest of the builds: what fits there fits everywhere
  if (prepare<128, 32, DEEP>(n_split) != cudaSuccess) { cudaGetLastError(); return 0; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_split);
  cfg.blockDim = dim3(NTD);
  cfg.dynamicSmemBytes = Lay<128, 32, DEEP>::OFF_MISC + sizeof(Misc<32>);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {(unsigned)n_split, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, decode_attn_kernel<128, 32, DEEP>, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}
int decode_clusters(int n_split, bool deep) { return deep ? clusters_t<true>(n_split) : clusters_t<false>(n_split); }

}  // namespace pc
