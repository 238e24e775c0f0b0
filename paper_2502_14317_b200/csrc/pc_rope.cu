// RoPE with position reuse (Sec. 3.1 "Parallel attention": positions restart in every
// chunk).  Pairs (t, t + d/2), angle p * theta^(-2t/d).  Queries and keys are rotated once,
// before the attention kernel, by a bandwidth-bound pass: the result is the fp64 rotation
// rounded once to bf16 (see pc_rope_exact.cuh for how fp32 arithmetic gets there), so rotated
// keys - an output that the gather copies - are reproducible to the bit.
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
  if (i == 0 && counter != nullptr) *counter = 0;           // work queue of the attention kernel that follows
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
// Outputs that the fp32 arithmetic cannot decide (about one in 1300) are redone exactly by the whole warp: the
// sixteen outputs of an undecided lane go to sixteen lanes, one each, and are patched into the row after the
// vector store.  (Handling them in the lane that found them would make a third of the warp's passes wait for one
// lane's slow path.)
//
// One launch takes one or two tensors of the same chunks and positions (keys and queries): grid.y first deals out the slices of
// the chunks of the first tensor, then those of the second.
//
// OWN_TABLE: a warp computes the table row of its position itself, in shared memory, before it waits for the kernel ahead
// (see launch_rope).
struct RopeAngles { double theta; int pos0; int *counter, *clear; };   // for OWN_TABLE; counter and clear (may be null) are set to 0
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
  if (OWN_TABLE && (blockIdx.x | blockIdx.y | blockIdx.z | threadIdx.x) == 0) {
    if (ang.counter != nullptr) *ang.counter = 0;
    if (ang.clear != nullptr) *ang.clear = 0;
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
  for (int c = slice; c < C; c += ny) {
    const uint16_t* src = x + (long long)c * s_chunk + (long long)p * s_tok + (long long)h_mine * s_head + g * 8;
    uint16_t* const dst_tok = y + ((size_t)c * L + p) * H * d;
    uint16_t* dst = dst_tok + (size_t)h_mine * d + g * 8;
    uint4 n1 = make_uint4(0, 0, 0, 0), n2 = make_uint4(0, 0, 0, 0);
    if (h_mine < H) {
      n1 = __ldg(reinterpret_cast<const uint4*>(src));
      n2 = __ldg(reinterpret_cast<const uint4*>(src + half));
    }
#pragma unroll 1
    for (int ps = blockIdx.z; ps < n_pass; ps += zs, src += step_src, dst += step_dst) {
      const bool active = h_first + ps * h_step < H;
      const uint4 x1 = n1, x2 = n2;
      if (ps + zs < n_pass && h_first + (ps + zs) * h_step < H) {                // the next pass's row is in flight during this one's arithmetic
        n1 = __ldg(reinterpret_cast<const uint4*>(src + step_src));
        n2 = __ldg(reinterpret_cast<const uint4*>(src + step_src + half));
      } else {
        n1 = make_uint4(0, 0, 0, 0); n2 = make_uint4(0, 0, 0, 0);
      }
      uint4 y1, y2;
      uint32_t amb = rope_two_pairs_fast(x1.x, x2.x, hi[0], y1.x, y2.x);
      amb |= rope_two_pairs_fast(x1.y, x2.y, hi[1], y1.y, y2.y);
      amb |= rope_two_pairs_fast(x1.z, x2.z, hi[2], y1.z, y2.z);
      amb |= rope_two_pairs_fast(x1.w, x2.w, hi[3], y1.w, y2.w);
      if (active) {
        *reinterpret_cast<uint4*>(dst) = y1;
        *reinterpret_cast<uint4*>(dst + half) = y2;
      }
      unsigned todo = __ballot_sync(0xFFFFFFFFu, active && amb != 0u);
      if (todo != 0u) {                                     // warp-uniform
        __syncwarp();                                       // the vector stores above precede the patches below
        const int t = (lane >> 1) & 7, second = lane & 1;   // lanes 0..15: pair t of the undecided lane, first / second output
        do {
          const int srcl = __ffs(todo) - 1;
          todo &= todo - 1;
          const uint32_t w1[4] = {__shfl_sync(0xFFFFFFFFu, x1.x, srcl), __shfl_sync(0xFFFFFFFFu, x1.y, srcl),
                                  __shfl_sync(0xFFFFFFFFu, x1.z, srcl), __shfl_sync(0xFFFFFFFFu, x1.w, srcl)};
          const uint32_t w2[4] = {__shfl_sync(0xFFFFFFFFu, x2.x, srcl), __shfl_sync(0xFFFFFFFFu, x2.y, srcl),
                                  __shfl_sync(0xFFFFFFFFu, x2.z, srcl), __shfl_sync(0xFFFFFFFFu, x2.w, srcl)};
          if (lane < 16) {
            const int wsel = t >> 1;
            const uint32_t u1 = wsel == 0 ? w1[0] : wsel == 1 ? w1[1] : wsel == 2 ? w1[2] : w1[3];
            const uint32_t u2 = wsel == 0 ? w2[0] : wsel == 1 ? w2[1] : wsel == 2 ? w2[2] : w2[3];
            const float a = __uint_as_float((t & 1) ? (u1 & 0xFFFF0000u) : (u1 << 16));
            const float b = __uint_as_float((t & 1) ? (u2 & 0xFFFF0000u) : (u2 << 16));
            const int sg = srcl % groups, sh = srcl / groups + ps * h_step;      // pair group and head of that lane
            const int pair = sg * 8 + t;
            const uint32_t r = second ? rope_one_exact<OWN_TABLE>(b, -a, pair, hi_row, lo_row, d_row)
                                      : rope_one_exact<OWN_TABLE>(a, b, pair, hi_row, lo_row, d_row);
            dst_tok[(size_t)sh * d + (second ? half : 0) + pair] = (uint16_t)r;
          }
        } while (todo != 0u);
        __syncwarp();
      }
    }
  }
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

void launch_rope(const RopeRows& a, const RopeRows* b, const RopeTable& tab, int C, int L, int d, double theta, int pos0,
                 int* counter, int* clear, cudaStream_t st) {
  const RopeTensor ta = rope_tensor(a, C, L, d);
  RopeTensor tb = {};
  if (b != nullptr) tb = rope_tensor(*b, C, L, d);
  const dim3 grid((unsigned)((L + 7) / 8), (unsigned)(ta.ny + tb.ny), (unsigned)(ta.nz > tb.nz ? ta.nz : tb.nz));
  const RopeAngles ang = {theta, pos0, counter, clear};
  // Up to 2 M values the warps compute their own table rows: one launch less, and the angles are found while the kernel ahead
  // still runs (us, table kernel / own rows; B x L x H x d: 1x64x32x128 5.2 / 3.8, 4x256x8x64 5.3 / 4.2, 1x1024x8x128
  // 7.3 / 5.5, 4x1024x8x64 8.1 / 7.7).  Above it, repeating the fp64 angles in every slice of the chunks and fewer free
  // registers cost more than the launch (16x64x32x128 9.9 / 10.4, 64x64x32x128 18.7 / 23.3, 4x8192x32x128 118 / 152).
  const long long values = (long long)C * L * d * (a.H + (b != nullptr ? b->H : 0));
  if (values <= (1 << 21)) {
    launch_chained(rope_rows_kernel<true>, grid, dim3(256), 0, st, 1, ta, tb, tab.hi, tab.lo, tab.exact, C, L, d, ang);
    return;
  }
  launch_chained(rope_table_kernel, dim3((unsigned)((L * (d / 4) + 255) / 256)), dim3(256), 0, st, 1, tab.exact, tab.hi, tab.lo, L, d / 2,
                 theta, pos0, counter, clear);
  launch_chained(rope_rows_kernel<false>, grid, dim3(256), 0, st, 1, ta, tb, tab.hi, tab.lo, tab.exact, C, L, d, ang);
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
