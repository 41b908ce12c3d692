// A CUDA runtime without a device for tests of the library's host code: allocations are host memory, launches are counted and do
// nothing, and launch number `fake_fail_at` (from 0) fails with an error that also stays pending, as the runtime's do.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <cstdlib>
#include <cstring>

static int launches = 0, fail_at = -1, early = 0;
static cudaError_t pending = cudaSuccess;
static thread_local struct { dim3 grid, block; size_t smem; void* stream; } cfg;

static cudaError_t launched() {
  if (launches++ != fail_at) return cudaSuccess;
  return pending = cudaErrorLaunchOutOfResources;
}
static CUresult encode_map(...) { return CUDA_SUCCESS; }

extern "C" {
void fake_fail_at(int k) { launches = 0; early = 0; fail_at = k; pending = cudaSuccess; }
int fake_launches() { return launches; }
int fake_early_launches() { return early; }              // launches that may start while the kernel before drains
int fake_pending_error() { return (int)pending; }

void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* stream) { cfg = {g, b, smem, stream}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* stream) {
  *g = cfg.grid; *b = cfg.block; *smem = cfg.smem; *(void**)stream = cfg.stream;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return launched(); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization && c->attrs[i].val.programmaticStreamSerializationAllowed) ++early;
  return launched();
}
cudaError_t cudaGetLastError() { const cudaError_t e = pending; pending = cudaSuccess; return e; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(1, n < 4096 ? n : 4096); return cudaSuccess; }   // (nothing runs on it)
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset2DAsync(void*, size_t, int, size_t, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo_v2(cudaStream_t, cudaStreamCaptureStatus* s, unsigned long long* id, cudaGraph_t*, const cudaGraphNode_t**, size_t*) {
  *s = cudaStreamCaptureStatusNone;
  if (id) *id = 0;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 148 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 233472 : 1024;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char word[64]; *p = word; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  *n = 120 / (int)c->attrs[0].val.clusterDim.x;          // (15 of eight, as on a B200)
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* found) {
  *fn = (void*)encode_map;
  if (found) *found = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
