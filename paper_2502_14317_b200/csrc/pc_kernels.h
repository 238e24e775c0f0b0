// Internal launcher declarations shared by the translation units of libpc.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

namespace pc {

// ---- pc_api.cu
// Every kernel launch of the library is counted here (see pc_launch_count in pc.h).
void note_launch();

// Launches of one call, and of calls on one stream, follow each other closely: every kernel is launched with programmatic
// stream serialisation, so that it is set up while its predecessor drains, and begins with chain() (kernels with a
// costly start after that start), which waits until everything before it on the stream has completed and then lets
// its successor be set up.  The successor is released AFTER the wait: at most two kernels overlap, so a kernel never
// shares an SM's L1 with a reader of the data that its predecessor replaces.
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, A... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void chain() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
}
#endif

// ---- pc_rope.cu
// Room for the cos/sin table of n_pos positions: exact[p * (d/2) + t] = (cos, sin)(  (pos0 + p) * theta^(-2t/d) ), fp64; hi, lo:
// the same entries split into an fp32 head and an fp32 tail (value = head + tail to 2^-48), one float4 per two pairs:
// (cos_2i, cos_2i+1, sin_2i, sin_2i+1).  Small inputs leave it unused.
struct RopeTable { double2* exact; float4 *hi, *lo; };
// y[c,p,h,:] = bf16( RoPE(x[c,p,h,:], position p) ), the fp64 rotation rounded once; x addressed by element strides
// (chunk, token, head), y contiguous [C,L,H,d].
struct RopeRows {
  const void* x;
  long long stride[3];
  void* y;
  int H;
};
// one tensor, or two (b not null) in the same launch; positions pos0 .. pos0 + L - 1; the COUNTER_WORDS
// of counter (pc_attn.h) and clear (each may be null) are set to 0
cudaError_t launch_rope(const RopeRows& a, const RopeRows* b, const RopeTable& tab, int C, int L, int d, double theta, int pos0,
                        int* counter, int* clear, cudaStream_t st);

// Per-chunk lengths: zero o[c, p, :, :], lse[c, :, p] and win_score[c, :, p] for p >= clamp(chunk_len[c], w + 1, L).
void launch_zero_chunk_tails(const int* chunk_len, int C, int L, int w, int Hq, int Hkv, int d, void* o,
                             const long long o_stride[3], float* lse, float* win_score, cudaStream_t st);

// ---- pc_select_gather.cu
void launch_chunk_score(const float* win_lse, int C, int n_per_chunk, float* score, cudaStream_t st);
void launch_select_chunks(const float* score, int C, int m, int lower_is_better, int* kept, cudaStream_t st);
// stand-in chunk score (as launch_chunk_score, same bits) followed by the chunk top-m, in one launch for C <= 64
void launch_score_select_chunks(const float* win_lse, int C, int n_per_chunk, int m, int lower_is_better, float* score,
                                int* kept, cudaStream_t st);
// attention calibration (Eq. 8): sizes of the sink and recency regions and the three thresholds; null = off
struct SelCalibArgs {
  int n_s, n_r;
  float lam_s, lam_m, lam_r;
};
cudaError_t launch_select_tokens(const float* win_score, const int* kept, int m, int Hkv, int L, int n_cand, int k,
                                 int* idx, const SelCalibArgs* calib, cudaStream_t st);
// online chunk queue: rank the chunks that move into a slot (slot_src[s] >= 0) and copy their kept rows into the slot
// storage, in one launch; cudaErrorNotSupported when k is too large for that (then rank and gather separately)
cudaError_t launch_select_gather_slots(const float* win_score, const int* slot_src, int m, int Hkv, int L, int n_cand,
                                       int k, const void* k_src, const void* v_src, const long long stride_elems[3],
                                       int d, void* q_k, void* q_v, int* q_pos, int sm_count, cudaStream_t st);
cudaError_t launch_gather_kv(const void* k_src, const void* v_src, const long long stride_elems[3], const int* kept,
                             const int* idx, int m, int Hkv, int k, int d, void* k_out, void* v_out, int* pos_out,
                             int sm_count, bool by_slot, cudaStream_t st);

// caches stored with room to grow: cache[b, hkv, Nk + i, :] = win[b, i, hkv, :] for the w new rows of every sequence
cudaError_t launch_append_kv(const void* k_win, const void* v_win, int B, int w, int Hkv, int d, long long Nk,
                             long long Nk_cap, void* k_cache, void* v_cache, cudaStream_t st);

// ---- pc_queue.cu (online chunk queue)
void launch_queue_init(float* q_score, int* q_chunk, int m, cudaStream_t st);
void launch_queue_update(const float* score, int Cb, int chunk_id0, int lower_is_better, int m, float* q_score,
                         int* q_chunk, int* slot_src, cudaStream_t st);
cudaError_t launch_queue_emit(const int* q_chunk, int m, int Hkv, int k, int d, const void* q_k, const void* q_v,
                              const int* q_pos, int* kept_out, int* slot_order, void* k_out, void* v_out,
                              int* pos_out, int sm_count, cudaStream_t st);

}  // namespace pc
