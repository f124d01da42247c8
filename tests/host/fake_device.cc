// Stand-ins for the CUDA runtime and for the kernel launchers, so that the host side of the library (csrc/wk_api.cu: argument
// checks and slot table) runs without a GPU.  "Device" memory is the caller's; the launchers do what matters to the slot table --
// the validity flags and poses -- and fail on request.
#include <string.h>

#include "wk_internal.cuh"

extern "C" {
int fail_compress = 0, fail_append = 0, fail_mark = 0;   // calls of that launcher fail while non-zero

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }

static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}

namespace wk {

int attention_partial_slots(int, int, int) { return 2; }
__nv_bfloat16* pool_rows(wk_ctx* ctx, __nv_bfloat16* base, int layer, int slot) {
  return base + (static_cast<int64_t>(layer) * ctx->cfg.pool_slots + slot) * ctx->C * ctx->D;
}
static wk_status set_slot(wk_ctx* ctx, int slot, int valid, const float* pose, int fail) {
  if (fail) return cuda_fail(ctx, cudaErrorLaunchOutOfResources);
  memcpy(ctx->poses_dev + slot * 8, pose, 8 * sizeof(float));
  ctx->valid_dev[slot] = valid;
  return WK_OK;
}
wk_status launch_compress(wk_ctx* ctx, const __nv_bfloat16*, int64_t, int, int32_t*, float*, cudaStream_t, AnchorStore*) {
  return fail_compress ? cuda_fail(ctx, cudaErrorLaunchOutOfResources) : WK_OK;
}
wk_status launch_append(wk_ctx* ctx, int, int, int slot, const __nv_bfloat16*, const __nv_bfloat16*, int64_t, const int32_t*,
                        cudaStream_t, const AnchorStore*, const float* mark_pose) {
  if (fail_append || mark_pose) return set_slot(ctx, slot, 1, mark_pose, fail_append);
  return WK_OK;
}
wk_status launch_slot_mark(wk_ctx* ctx, int slot, int valid, const float* pose, cudaStream_t) {
  return set_slot(ctx, slot, valid, pose, fail_mark);
}
wk_status launch_retrieve(wk_ctx*, const float*, int, int32_t*, double*, cudaStream_t) { return WK_OK; }
wk_status launch_retrieve_query(wk_ctx*, int, const __nv_bfloat16*, int, int, int32_t*, float*, cudaStream_t) { return WK_OK; }
size_t retrieve_scan_scratch_bytes() { return 16; }
wk_status launch_retrieve_scan(wk_ctx*, const float*, const int32_t*, int64_t, const float*, int, int32_t*, double*, int, void*,
                               cudaStream_t) { return WK_OK; }
wk_status launch_attention(wk_ctx*, int, const __nv_bfloat16*, int, const wk_dense_seg*, int, const int32_t*, int, __nv_bfloat16*,
                           float*, int, cudaStream_t, bool) { return WK_OK; }

}  // namespace wk
