// Parameter blocks and launchers of the attention kernels (internal).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace pc {

// Words that follow a work counter, zeroed with it: blocks with window rows that are done, by (chunk, kv-head) group.
constexpr int COUNTER_WORDS = 64, MAX_SPREAD_GROUPS = COUNTER_WORDS - 1;

struct PrefillParams {
  int C, L, w, Hq, Hkv;
  float scale_log2;              // softmax scale * log2(e)
  const int* chunk_len;          // [C] tokens per chunk (window included) or null: all L
  float* lse;                    // [C,Hq,L] or null
  float* win_lse;                // [C,Hq,w], or null: win_lse2 is converted afterwards (launch_win_lse_natural)
  float* win_lse2;               // [C,Hq,w] in log2 units, as the score sweep needs it
  float* win_score;              // [C,Hkv,L]
  int* status;                   // device status word or null
  int* counter;                  // work-queue counter and COUNTER_WORDS - 1 words behind it, zeroed before launch
  int sweep_slices;              // 0: a group's score sweep belongs to its tail item; n: it is n items of its own (few groups)
  int wait_kcycles;              // limit of every device-side wait, in units of 1024 cycles
  int skip_final_publication;    // test hook of the bounded waits (see pc_debug_bounded_wait_test in pc.h)
};

// maps: rotated q (box 64 x 1 x 128 tokens), k_rot, v, o (store), rotated q with a wp-row box, k_rot with a 64-token box
cudaError_t launch_prefill_attn(const CUtensorMap* maps, const PrefillParams& prm, int d, int sm_count, cudaStream_t st);

// x[i] *= ln 2: log-sum-exp in log2 units to natural ones
cudaError_t launch_win_lse_natural(float* x, long long n, cudaStream_t st);

// Parallel attention, more than 32 query rows per kv-head (pc_parallel.cu).
struct ParallelParams {
  int B, w, Hq, Hkv, Nk;
  int alt;                       // 1: the two blocks of a CTA hold the same rows and take alternate key tiles; 0: they hold
                                 // different rows and share the tiles
  int n_rg;                      // row groups per kv-head (128 rows per CTA with alt, else 256; twice that on CTA pairs)
  int n_cache_tiles, n_split;    // 128-key tiles of the cache; key splits (over those tiles and the window's own)
  float scale_log2;
  float* part_o;                 // [B,Hq,n_split,w,d] fp32 unnormalised partial outputs (n_split > 1)
  float* part_ml;                // [B,Hq,n_split,w,2] (running max in log2 units, sum)
  __nv_bfloat16* out;            // [B,w,Hq,d]
  float* lse_out;                // [B,Hq,w] or null
  int* status;
  int* counter;                  // work-queue counter, zeroed before launch
  int wait_kcycles;              // limit of every device-side wait, in units of 1024 cycles
  int skip_final_publication;    // test hook of the bounded waits (see pc_debug_bounded_wait_test in pc.h)
};
// maps: rotated q_win (w-row box), k_cache (128-key box; pair: 64), v_cache (128), k_win (128-row box over w tokens; pair:
// 64), v_win (128)
cudaError_t launch_parallel_attn(const CUtensorMap* maps, const ParallelParams& prm, int d, bool pair, int sm_count, cudaStream_t st);

// Parallel attention for few query rows (pc_decode.cu): Hq / Hkv * w <= 32.  One launch, no workspace.
struct DecodeParams {
  int B, w, Hq, Hkv, Nk;
  int n_cache_tiles, n_split;    // 128-key tiles of the cache; CTAs (of a cluster) per (sequence, kv-head), 1 .. 16
  int deep;                      // head size 128: six stages and one CTA per SM, not three and two
  int q_pos0;
  float rope_theta, scale_log2;
  const void *q_win, *k_win, *v_win;
  void *k_append, *v_append;     // caches to append the new entries to at Nk (rows Nk_cap apart), or null
  long long Nk_cap;
  __nv_bfloat16* out;            // [B,w,Hq,d]
  float* lse_out;                // [B,Hq,w] or null
  int* status;
  int wait_kcycles;
};
// maps: k_cache, v_cache (128-key box), k_win, v_win (128-row box over w tokens)
cudaError_t launch_decode_attn(const CUtensorMap* maps, const DecodeParams& prm, int d, cudaStream_t st);
// clusters of n_split CTAs that the current device runs at a time
int decode_clusters(int n_split, bool deep);

}  // namespace pc
