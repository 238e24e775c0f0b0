// RoPE with position reuse (Sec. 3.1 "Parallel attention": positions restart in every
// chunk).  Pairs (t, t + d/2), angle p * theta^(-2t/d).  Queries and keys are rotated once,
// before the attention kernel, by a bandwidth-bound pass: the result is the fp64 rotation
// rounded once to bf16 (see pc_rope_exact.cuh for how fp32 arithmetic gets there), so rotated
// keys - an output that the gather copies - are reproducible to the bit.
#include "pc_attn.h"
#include "pc_kernels.h"
#include "pc_rope_exact.cuh"

namespace pc {

__device__ __forceinline__ void rope_angle(double theta, int half, int pos, int t, double& c, double& s) {
  const double inv_freq = pow(theta, -2.0 * (double)t / (double)(2 * half));
  sincos((double)pos * inv_freq, &s, &c);
}

// tab: (cos, sin) per (position, pair), fp64.  tab_hi / tab_lo: fp32 heads / tails of the same values, one float4
// per two consecutive pairs (cos_2i, cos_2i+1, sin_2i, sin_2i+1); value = head + tail to 2^-48.
__global__ void rope_table_kernel(double2* __restrict__ tab, float4* __restrict__ tab_hi, float4* __restrict__ tab_lo, int n_pos,
                                  int half, double theta, int pos0, int* __restrict__ counter, int* __restrict__ clear) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;      // one thread per two pairs
  const int p = i / (half / 2), t = 2 * (i % (half / 2));
  const bool mine = i < n_pos * (half / 2);
  double c[2], s[2];
  if (mine) {
#pragma unroll
    for (int e = 0; e < 2; ++e) rope_angle(theta, half, pos0 + p, t + e, c[e], s[e]);
  }
  chain();                                                  // the arithmetic needs nothing from before; the tables may still be in use
  if (i < COUNTER_WORDS && counter != nullptr) counter[i] = 0;   // work queue of the attention kernel that follows
  if (i == 0 && clear != nullptr) *clear = 0;
  if (!mine) return;
  for (int e = 0; e < 2; ++e) tab[(size_t)p * half + t + e] = make_double2(c[e], s[e]);
  const float c0 = (float)c[0], c1 = (float)c[1], s0 = (float)s[0], s1 = (float)s[1];
  tab_hi[i] = make_float4(c0, c1, s0, s1);
  tab_lo[i] = make_float4((float)(c[0] - (double)c0), (float)(c[1] - (double)c1), (float)(s[0] - (double)s0), (float)(s[1] - (double)s1));
}

// y[c,p,h,:] = bf16( RoPE(x[c,p,h,:], position p) ).  One warp owns one position: a lane holds 8 consecutive
// pairs (t .. t+7) and takes every (32 / (d/16))-th head, so one pass of the warp reads and writes a contiguous
// piece of the token's row (1 KB for d = 128), and a block of 8 warps streams 8 adjacent rows: the DRAM pages
// are walked front to back, as a copy would.  The table entries of (position, pairs) stay in registers across
// the heads and across the chunks of the block's slice.
// Outputs that the fp32 arithmetic cannot decide (about one in 1300, so something in a third of a warp's passes) are redone
// exactly: a lane that has any leaves its sixteen inputs in a list of the warp, and whenever there are two such lanes
// on the list their thirty-two outputs go to the thirty-two lanes and are patched into the rows.  (One lane at a time, its
// inputs spread by shuffles: a third of all instructions; 4 x 8192 x 32 x 128, inputs not yet through the ring below, 117 us for 110.)
//
// One launch takes one or two tensors of the same chunks and positions (keys and queries): grid.y first deals out the slices of
// the chunks of the first tensor, then those of the second.
//
// OWN_TABLE: a warp computes the table row of its position itself, in shared memory, before it waits for the kernel ahead
// (see launch_rope).
struct RopeAngles { double theta; int pos0; int *counter, *clear; };   // for OWN_TABLE; counter and clear (may be null) are set to 0
__device__ __forceinline__ void copy_async16(void* smem_dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }
struct RopeTodo { uint4 x1, x2; uint16_t* dst; int g; };       // a lane's inputs, where its outputs go, its group of pairs
struct RopeRow { float4 hi[32], lo[32]; double2 exact[64]; };
struct RopeTensor {
  const uint16_t* x;
  uint16_t* y;
  long long s_chunk, s_tok, s_head;                         // element strides of x; y is contiguous
  int H, ny, nz;                                            // heads; slices of the chunks; parts of the head passes
};
template <bool OWN_TABLE>
__global__ void __launch_bounds__(256, 4) rope_rows_kernel(const __grid_constant__ RopeTensor ta, const __grid_constant__ RopeTensor tb,
                                                           const float4* __restrict__ tab_hi, const float4* __restrict__ tab_lo,
                                                           const double2* __restrict__ tab, int C, int L, int d, RopeAngles ang) {
  __shared__ RopeRow own[OWN_TABLE ? 8 : 1];
  const int half = d / 2, lane = threadIdx.x & 31;
  const int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  RopeRow& row = own[OWN_TABLE ? threadIdx.x >> 5 : 0];
  __shared__ RopeTodo todo_lists[8][33];
  RopeTodo* const todo = todo_lists[threadIdx.x >> 5];
  int n_todo = 0;                                           // the same in all lanes
  if (OWN_TABLE && p < L) {
    for (int t = lane; t < half; t += 32) {
      double2 e;
      rope_angle(ang.theta, half, ang.pos0 + p, t, e.x, e.y);
      const float c0 = (float)e.x, s0 = (float)e.y;
      float* const hi = reinterpret_cast<float*>(&row.hi[t >> 1]) + (t & 1);
      float* const lo = reinterpret_cast<float*>(&row.lo[t >> 1]) + (t & 1);
      hi[0] = c0; hi[2] = s0;
      lo[0] = (float)(e.x - (double)c0); lo[2] = (float)(e.y - (double)s0);
      row.exact[t] = e;
    }
    __syncwarp();
  }
  chain();
  if (OWN_TABLE && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) {
    if (ang.counter != nullptr && threadIdx.x < COUNTER_WORDS) ang.counter[threadIdx.x] = 0;
    if (ang.clear != nullptr && threadIdx.x == 0) *ang.clear = 0;
  }
  const bool second_tensor = (int)blockIdx.y >= ta.ny;      // the same for the whole block
  const uint16_t* __restrict__ const x = second_tensor ? tb.x : ta.x;
  uint16_t* __restrict__ const y = second_tensor ? tb.y : ta.y;
  const long long s_chunk = second_tensor ? tb.s_chunk : ta.s_chunk, s_tok = second_tensor ? tb.s_tok : ta.s_tok,
                  s_head = second_tensor ? tb.s_head : ta.s_head;
  const int H = second_tensor ? tb.H : ta.H, ny = second_tensor ? tb.ny : ta.ny, zs = second_tensor ? tb.nz : ta.nz;
  const int slice = second_tensor ? (int)blockIdx.y - ta.ny : (int)blockIdx.y;
  if ((int)blockIdx.z >= zs) return;
  const int groups = half / 8;                              // 16-byte groups per half row (4 or 8)
  if (p >= L) return;                                       // whole warps leave together
  const int g = lane % groups, h_first = lane / groups, h_step = 32 / groups;
  const size_t row0 = (size_t)p * half;                     // first pair of this position in the tables
  const float4* hi_row = OWN_TABLE ? row.hi : tab_hi + row0 / 2;
  const float4* lo_row = OWN_TABLE ? row.lo : tab_lo + row0 / 2;
  const double2* d_row = OWN_TABLE ? row.exact : tab + row0;
  float4 hi[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) hi[i] = table_entry<OWN_TABLE>(hi_row + g * 4 + i);
  // small inputs: the head passes are dealt out over grid.z (zs parts)
  const long long step_src = (long long)h_step * zs * s_head;
  const size_t step_dst = (size_t)h_step * zs * d;
  const int n_pass = (H + h_step - 1) / h_step;
  const int h_mine = h_first + (int)blockIdx.z * h_step;    // this thread's head in its first pass
  // outputs of entries i and i + 1 (an entry below 0 is none)
  auto redo = [&](int i) {
    __syncwarp();                                           // the list, and the vector stores that the patches follow
    const int t = (lane >> 1) & 7, second = lane & 1, e = i + (lane >> 4);
    if (e >= 0) {
      const RopeTodo& d = todo[e];
      const float a = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(&d.x1)[t] << 16);
      const float b = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(&d.x2)[t] << 16);
      const int pair = d.g * 8 + t;
      const uint32_t r = second ? rope_one_exact<OWN_TABLE>(b, -a, pair, hi_row, lo_row, d_row)
                                : rope_one_exact<OWN_TABLE>(a, b, pair, hi_row, lo_row, d_row);
      d.dst[(second ? half : 0) + t] = (uint16_t)r;
    }
    __syncwarp();
  };
  // A lane's inputs of the next passes come through a ring in shared memory (its own slots only: nothing to synchronise), so that
  // DEPTH - 1 passes are in flight; with one in registers the pass was bound by the latency of memory (4 x 8192 x 32 x 128: 110
  // us, 97 with two or three passes in the ring, 83 at the copy bandwidth; 16 x 8192 x 8 x 128: 116 and 100).
  constexpr int DEPTH = OWN_TABLE ? 2 : 3;
  __shared__ uint4 ring[8][DEPTH][2][32];
  uint4(*const mine)[2][32] = ring[threadIdx.x >> 5];
  int c_next = slice, ps_next = blockIdx.z;
  const uint16_t* src = x + (long long)slice * s_chunk + (long long)p * s_tok + (long long)h_mine * s_head + g * 8;
  auto fetch = [&](int slot) {
    if (c_next < C) {
      if (h_first + ps_next * h_step < H) {                 // (lanes without a row compute on what is there and store nothing)
        copy_async16(&mine[slot][0][lane], src);
        copy_async16(&mine[slot][1][lane], src + half);
      }
      ps_next += zs;
      src += step_src;
      if (ps_next >= n_pass) {
        ps_next = blockIdx.z;
        c_next += ny;
        src = x + (long long)c_next * s_chunk + (long long)p * s_tok + (long long)h_mine * s_head + g * 8;
      }
    }
    copy_async_commit();
  };
#pragma unroll
  for (int i = 0; i < DEPTH - 1; ++i) fetch(i);
  int slot = 0;
  for (int c = slice; c < C; c += ny) {
    uint16_t* dst = y + ((size_t)c * L + p) * H * d + (size_t)h_mine * d + g * 8;
#pragma unroll 1
    for (int ps = blockIdx.z; ps < n_pass; ps += zs, dst += step_dst) {
      const bool active = h_first + ps * h_step < H;
      fetch((slot + DEPTH - 1) % DEPTH);
      copy_async_wait<DEPTH - 1>();
      const uint4 x1 = mine[slot][0][lane], x2 = mine[slot][1][lane];
      slot = (slot + 1) % DEPTH;
      uint4 y1, y2;
      uint32_t amb = rope_two_pairs_fast(x1.x, x2.x, hi[0], y1.x, y2.x);
      amb |= rope_two_pairs_fast(x1.y, x2.y, hi[1], y1.y, y2.y);
      amb |= rope_two_pairs_fast(x1.z, x2.z, hi[2], y1.z, y2.z);
      amb |= rope_two_pairs_fast(x1.w, x2.w, hi[3], y1.w, y2.w);
      if (active) {
        *reinterpret_cast<uint4*>(dst) = y1;
        *reinterpret_cast<uint4*>(dst + half) = y2;
      }
      const unsigned undecided = __ballot_sync(0xFFFFFFFFu, active && amb != 0u);
      if (undecided != 0u) {                                // warp-uniform
        if ((undecided >> lane) & 1u) todo[n_todo + __popc(undecided & ((1u << lane) - 1u))] = {x1, x2, dst, g};
        n_todo += __popc(undecided);
        for (; n_todo >= 2; n_todo -= 2) redo(n_todo - 2);
      }
    }
  }
  if (n_todo != 0) redo(n_todo - 2);
}

static RopeTensor rope_tensor(const RopeRows& r, int C, int L, int d) {
  RopeTensor t;
  t.x = (const uint16_t*)r.x; t.y = (uint16_t*)r.y;
  t.s_chunk = r.stride[0]; t.s_tok = r.stride[1]; t.s_head = r.stride[2];
  t.H = r.H;
  const int bx = (L + 7) / 8;                               // 8 positions per block
  // a slice of the chunks per block: the table entries are reused over the slice; enough blocks to fill the GPU
  t.ny = (4736 + bx - 1) / bx;
  t.ny = t.ny < 1 ? 1 : (t.ny > C ? C : t.ny);
  // a few positions and chunks only (the query window of one sequence): the passes over the heads, which a warp
  // would otherwise walk one after the other, become blocks of their own
  const int n_pass = (r.H + 32 / (d / 16) - 1) / (32 / (d / 16));
  t.nz = bx * t.ny < 592 ? 592 / (bx * t.ny) : 1;
  t.nz = t.nz > n_pass ? n_pass : (t.nz < 1 ? 1 : t.nz);
  return t;
}

cudaError_t launch_rope(const RopeRows& a, const RopeRows* b, const RopeTable& tab, int C, int L, int d, double theta, int pos0,
                        int* counter, int* clear, cudaStream_t st) {
  const RopeTensor ta = rope_tensor(a, C, L, d);
  RopeTensor tb = {};
  if (b != nullptr) tb = rope_tensor(*b, C, L, d);
  const dim3 grid((unsigned)((L + 7) / 8), (unsigned)(ta.ny + tb.ny), (unsigned)(ta.nz > tb.nz ? ta.nz : tb.nz));
  const RopeAngles ang = {theta, pos0, counter, clear};
  // Up to 1 M values the warps compute their own table rows: one launch less, and the angles are found while the kernel ahead
  // still runs (us, table kernel / own rows; C x L x H x d: 1x64x32x128 4.1 / 2.8, 4x256x8x64 4.2 / 2.9, 1x1024x8x128
  // 5.5 / 4.8, 4x64x32x128 4.7 / 5.1 and 2 us less host time).  Above it, repeating the fp64 angles in every slice of the
  // chunks and fewer free registers cost more than the launch (8x64x32x128 5.7 / 6.8, 64x64x32x128 14.7 / 18.1, 4x8192x32x128
  // 97 / 129).
  const long long values = (long long)C * L * d * (a.H + (b != nullptr ? b->H : 0));
  if (values <= (1 << 20))
    return launch_chained(rope_rows_kernel<true>, grid, dim3(256), 0, st, 1, ta, tb, tab.hi, tab.lo, tab.exact, C, L, d, ang);
  if (cudaError_t e = launch_chained(rope_table_kernel, dim3((unsigned)((L * (d / 4) + 255) / 256)), dim3(256), 0, st, 1, tab.exact, tab.hi,
                                     tab.lo, L, d / 2, theta, pos0, counter, clear);
      e != cudaSuccess) return e;
  return launch_chained(rope_rows_kernel<false>, grid, dim3(256), 0, st, 1, ta, tb, tab.hi, tab.lo, tab.exact, C, L, d, ang);
}

// Rows behind the end of a chunk that is shorter than L (per-chunk lengths): outputs read as zero there.
__global__ void zero_chunk_tails_kernel(const int* __restrict__ chunk_len, int L, int w, int Hq, int Hkv, int d,
                                        uint16_t* __restrict__ o, long long so_chunk, long long so_tok, long long so_head,
                                        float* __restrict__ lse, float* __restrict__ win_score) {
  chain();
  const int c = blockIdx.y;
  int len = chunk_len[c];
  len = len > L ? L : (len <= w ? w + 1 : len);
  const int n_tail = L - len;
  const long long per_tok = (long long)Hq * (d / 8);        // 16-byte pieces of an output row over all heads
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)n_tail * per_tok;
       i += (long long)gridDim.x * blockDim.x) {
    const int p = len + (int)(i / per_tok), rest = (int)(i % per_tok), h = rest / (d / 8), piece = rest % (d / 8);
    *reinterpret_cast<uint4*>(o + (long long)c * so_chunk + (long long)p * so_tok + (long long)h * so_head + piece * 8) =
        make_uint4(0, 0, 0, 0);
  }
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)n_tail * (Hq + Hkv);
       i += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(i / n_tail), p = len + (int)(i % n_tail);
    if (row < Hq) { if (lse != nullptr) lse[((size_t)c * Hq + row) * L + p] = 0.0f; }
    else win_score[((size_t)c * Hkv + (row - Hq)) * L + p] = 0.0f;
  }
}

void launch_zero_chunk_tails(const int* chunk_len, int C, int L, int w, int Hq, int Hkv, int d, void* o,
                             const long long o_stride[3], float* lse, float* win_score, cudaStream_t st) {
  launch_chained(zero_chunk_tails_kernel, dim3(64, (unsigned)C), dim3(256), 0, st, 1, chunk_len, L, w, Hq, Hkv, d, (uint16_t*)o, o_stride[0],
                                                                o_stride[1], o_stride[2], lse, win_score);
}

}  // namespace pc
