// Softmax of one key tile, shared by the chunk-local attention kernels (thread = query row = TMEM lane).
#pragma once
#include "pc_sm100.cuh"

namespace pc {

constexpr float LAZY_RESCALE_LOG2 = 8.0f;      // the reference maximum is raised only when it grows by more than 2^8
constexpr float MAX_HALF_SUM = 256.0f;         // 2^8, see softmax_tile
// All exponentials run on the MUFU pipe (ex2), 1024 cycles a tile and warp.  Evaluating every fourth pair as a polynomial on
// the FMA pipe took a seventh off a tile's cycles and made every workload slower: these kernels run at the board's
// power cap, and twenty FMA-pipe instructions cost more energy than the two ex2 they replace (with an S of each block and one
// issuing thread: 128K tokens, 32/8 heads 9244 us with every fourth pair, 8946 with every eighth, 8725 with none; head size 64
// at 32K tokens 1018, 977, 953).

__device__ __forceinline__ uint64_t dup2(float v) { return pack_f32x2(v, v); }

// 32 logits -> 16 packed bf16 pairs; partial sums in sum2
__device__ __forceinline__ void exps32(const uint32_t (&s)[32], uint64_t scale2, uint64_t negm2, uint64_t (&sum2)[2],
                                       uint32_t (&packed)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), scale2, negm2);
    float x0, x1;
    unpack_f32x2(x2, x0, x1);
    const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
    sum2[i & 1] = add_f32x2(sum2[i & 1], pack_f32x2(p0, p1));
    packed[i] = pack_bf16x2(p0, p1);
  }
}
__device__ __forceinline__ float max32(const uint32_t (&s)[32]) {
  float a = fmax3(__uint_as_float(s[0]), __uint_as_float(s[1]), __uint_as_float(s[2]));
#pragma unroll
  for (int j = 3; j < 31; j += 2) a = fmax3(a, __uint_as_float(s[j]), __uint_as_float(s[j + 1]));
  return fmaxf(a, __uint_as_float(s[31]));
}
// masked columns (>= vis) of a 32-column piece whose first column is `col0`
__device__ __forceinline__ void mask32(uint32_t (&s)[32], int col0, int vis) {
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (col0 + j >= vis) s[j] = 0xFF800000u;                       // -inf
}
// after tmem_wait_ld: ties the loaded registers to the wait, so that no use of them moves above it
__device__ __forceinline__ void loaded(uint32_t (&r)[32]) {
#pragma unroll
  for (int i = 0; i < 32; i += 8)
    asm volatile("" : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]), "+r"(r[i + 5]), "+r"(r[i + 6]), "+r"(r[i + 7]));
}

struct RowState { float m, l; };               // reference maximum (log2 units) of a row and its sum relative to that

// multiplies the accumulator rows of this warp by alpha
template <int D>
__device__ __forceinline__ void rescale_rows(uint32_t o_taddr, float alpha) {
#pragma unroll 1
  for (int q = 0; q < D / 8; ++q) {
    uint32_t o[8];
    tmem_ld8(o_taddr + q * 8, o);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
    tmem_st8(o_taddr + q * 8, o);
  }
}

// One 128-key tile.  The logits are taken into registers at once and their columns given back (on_read), so that the next
// logits are computed meanwhile.  The exponentials of the first 64 keys are taken against the reference maximum of the tiles BEFORE
// this one and published only when none of them, and no logit of the other half, exceeds it by more than 2^8 in any row of the
// warp (otherwise the reference is raised to the maximum, the accumulator rescaled and the first half repeated).  Of the first
// half the sum tells, which is needed anyway: while it is at most 2^8, so is every term; if it is more, or no number, the
// maximum is looked up.  Of the other half the maximum is found beside the exponentials.  (With the maximum of both halves, in
// a loop, one issuing thread: 128K tokens, 32/8 heads 7894 -> 7839 us, 32/32 heads 5307 -> 5265, head size 64, 32K tokens
// 886 -> 874.  The second half by its sum as well, with a barrier for the first half's P V: 7842, 5283, 888.)
// GEN: tiles with masked columns (columns >= vis; vis <= 0: all) and the first tile of a block; the tiles between
// run straight-line code (the branches around the masks cost 300 of 1240 cycles).
// Hooks: on_read() - all logits are in registers; before_p() - called before the accumulator is touched and before
// probabilities are stored at p_taddr (64 columns); on_half(), on_full() - keys 0..63 / all keys of P are in TMEM.
template <int D, bool GEN, class Hooks>
__device__ __forceinline__ void softmax_tile(uint32_t s_taddr, uint32_t p_taddr, uint32_t o_taddr, int vis, bool first_tile,
                                             float scale_log2, RowState& st, const Hooks& hk) {
  const uint64_t scale2 = dup2(scale_log2);
  uint64_t sum2[2] = {0ull, 0ull};
  uint32_t pk[16], c0[32], c1[32], c2[32], c3[32];
  tmem_ld32(s_taddr, c0);
  tmem_ld32(s_taddr + 32, c1);
  tmem_ld32(s_taddr + 64, c2);
  tmem_ld32(s_taddr + 96, c3);
  tmem_wait_ld();
  loaded(c0); loaded(c1); loaded(c2); loaded(c3);
  hk.on_read();
  if (GEN) { mask32(c0, 0, vis); mask32(c1, 32, vis); mask32(c2, 64, vis); mask32(c3, 96, vis); }
  auto first_half = [&]() {
    const uint64_t negm2 = dup2(st.m == -INFINITY ? 0.0f : -st.m);  // nothing visible so far: exp2(-inf) = 0
    exps32(c0, scale2, negm2, sum2, pk);
    tmem_st16(p_taddr, pk);
    exps32(c1, scale2, negm2, sum2, pk);
    tmem_st16(p_taddr + 16, pk);
  };
  hk.before_p();
  float a0, a1, half_sum = 0.0f;
  bool raise = GEN && first_tile;
  if (!GEN || !first_tile) {
    first_half();
    unpack_f32x2(add_f32x2(sum2[0], sum2[1]), a0, a1);
    half_sum = a0 + a1;
    raise = !(half_sum <= (st.m == -INFINITY ? -1.0f : MAX_HALF_SUM));
  }
  raise |= fmaxf(max32(c2), max32(c3)) * scale_log2 > st.m + LAZY_RESCALE_LOG2;
  if (__any_sync(0xFFFFFFFFu, raise)) {                            // rare; warp-uniform: each warp owns its 32 lanes of O
    const float mx = fmaxf(fmaxf(max32(c0), max32(c1)), fmaxf(max32(c2), max32(c3))) * scale_log2;
    float alpha = 1.0f;
    if (raise) {
      const float m_new = fmaxf(st.m, mx);
      alpha = (st.m == -INFINITY) ? 0.0f : fast_exp2(st.m - m_new);
      st.m = m_new;
      st.l *= alpha;
    }
    if (!GEN || !first_tile) {
      rescale_rows<D>(o_taddr, alpha);
      tmem_wait_st();                                              // the first half is about to be stored again
    }
    sum2[0] = sum2[1] = 0ull;
    first_half();
    unpack_f32x2(add_f32x2(sum2[0], sum2[1]), a0, a1);
    half_sum = a0 + a1;
  }
  tmem_wait_st();
  hk.on_half();
  st.l += half_sum;
  sum2[0] = sum2[1] = 0ull;
  const uint64_t negm2 = dup2(st.m == -INFINITY ? 0.0f : -st.m);
  exps32(c2, scale2, negm2, sum2, pk);
  tmem_st16(p_taddr + 32, pk);
  exps32(c3, scale2, negm2, sum2, pk);
  tmem_st16(p_taddr + 48, pk);
  tmem_wait_st();
  hk.on_full();
  unpack_f32x2(add_f32x2(sum2[0], sum2[1]), a0, a1);
  st.l += a0 + a1;
}

}  // namespace pc
