// A CUDA runtime and the other launchers of libpc as counters, linked with pc_api.cu and pc_rope.cu into a library that runs without a
// GPU: host code of the C ABI with launches that can be made to fail.
#include <cuda.h>
#include <cuda_runtime.h>
#include "pc_attn.h"
#include "pc_kernels.h"

static int g_fail_at = -1, g_launches = 0, g_attention = 0, g_items = 0, g_grid = 0;
static cudaError_t g_last = cudaSuccess;

extern "C" {
__attribute__((visibility("default"))) void fake_reset(int fail_at) { g_fail_at = fail_at; g_launches = g_attention = 0; g_last = cudaSuccess; }
__attribute__((visibility("default"))) int fake_attention_launches() { return g_attention; }
__attribute__((visibility("default"))) int fake_window_items() { return g_items; }
__attribute__((visibility("default"))) int fake_last_grid() { return g_grid; }
__attribute__((visibility("default"))) int fake_last_error() { return (int)g_last; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = (void*)(1 << 20); return cudaSuccess; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  g_grid = (int)c->gridDim.x;
  return g_launches++ == g_fail_at ? (g_last = cudaErrorLaunchOutOfResources) : cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrMultiProcessorCount ? 148 : 10; return cudaSuccess; }
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                       const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* r) {
  *fn = (void*)encode; *r = cudaDriverEntryPointSuccess; return cudaSuccess;
}
}

namespace pc {
static cudaError_t attention() {                                  // (the real ones launch through the runtime too)
  ++g_attention;
  return g_launches++ == g_fail_at ? (g_last = cudaErrorLaunchOutOfResources) : cudaSuccess;
}
cudaError_t launch_prefill_attn(const CUtensorMap*, const PrefillParams&, int, int, cudaStream_t) { return attention(); }
cudaError_t launch_parallel_attn(const CUtensorMap*, const ParallelParams& p, int, bool, int, cudaStream_t) {
  g_items = p.B * p.Hkv * p.n_rg * p.n_split;
  return attention();
}
cudaError_t launch_decode_attn(const CUtensorMap*, const DecodeParams&, int, cudaStream_t) { return attention(); }
cudaError_t launch_win_lse_natural(float*, long long, cudaStream_t) { return cudaSuccess; }
int decode_clusters(int, bool) { return 8; }
// (the ranking and the gather may be linked too)
__attribute__((weak)) void launch_chunk_score(const float*, int, int, float*, cudaStream_t) {}
__attribute__((weak)) void launch_select_chunks(const float*, int, int, int, int*, cudaStream_t) {}
__attribute__((weak)) void launch_score_select_chunks(const float*, int, int, int, int, float*, int*, cudaStream_t) {}
__attribute__((weak)) cudaError_t launch_select_tokens(const float*, const int*, int, int, int, int, int, int*, const SelCalibArgs*, cudaStream_t) { return cudaSuccess; }
__attribute__((weak)) cudaError_t launch_select_gather_slots(const float*, const int*, int, int, int, int, int, const void*, const void*, const long long*, int, void*,
                                       void*, int*, int, cudaStream_t) { return cudaSuccess; }
__attribute__((weak)) cudaError_t launch_gather_kv(const void*, const void*, const long long*, const int*, const int*, int, int, int, int, void*, void*, int*, int, bool,
                             cudaStream_t) { return cudaSuccess; }
__attribute__((weak)) cudaError_t launch_append_kv(const void*, const void*, int, int, int, int, long long, long long, void*, void*, cudaStream_t) { return cudaSuccess; }
void launch_queue_init(float*, int*, int, cudaStream_t) {}
void launch_queue_update(const float*, int, int, int, int, float*, int*, int*, cudaStream_t) {}
cudaError_t launch_queue_emit(const int*, int, int, int, int, const void*, const void*, const int*, int*, int*, void*, void*, int*, int, cudaStream_t) {
  return cudaSuccess;
}
}  // namespace pc
