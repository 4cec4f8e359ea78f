// Stand-in for the CUDA runtime and the kernel launchers under the host side
// of the C ABI (evisel_capi.cpp), so that its bookkeeping and error paths run
// without a GPU: device memory is host memory, copies are immediate, a launch
// is counted by name, and the named call can be made to fail once.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include <cuda.h>
#include <cuda_runtime.h>

#include "evisel_internal.h"

namespace {

std::map<std::string, int> g_calls;
std::string g_fail_name;      // this call fails ...
int g_fail_after = 0;         // ... after as many that succeed

cudaError_t call(const char* name) {
  ++g_calls[name];
  if (g_fail_name == name && g_fail_after-- == 0) {
    g_fail_name.clear();
    return cudaErrorMemoryAllocation;
  }
  return cudaSuccess;
}

cudaError_t allocate(void** p, size_t n, const char* name) {
  const cudaError_t e = call(name);
  if (e == cudaSuccess) *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
  return e;
}

CUresult encode(CUtensorMap* map, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  std::memset(map, 0, sizeof(*map));
  return call("encode") == cudaSuccess ? CUDA_SUCCESS : CUDA_ERROR_INVALID_VALUE;
}

}  // namespace

extern "C" {

void fake_fail(const char* name, int after) {
  g_fail_name = name;
  g_fail_after = after;
}
int fake_calls(const char* name) { return g_calls[name]; }

cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n, "cudaMalloc"); }
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n, "cudaMallocHost"); }
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return call("cudaMemset"); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return call("cudaMemsetAsync"); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  return std::memcpy(d, s, n), call("cudaMemcpy");
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return std::memcpy(d, s, n), call("cudaMemcpyAsync");
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = reinterpret_cast<cudaEvent_t>(1);
  return call("cudaEventCreateWithFlags");
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return call("cudaEventRecord"); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return call("cudaStreamWaitEvent"); }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *p = reinterpret_cast<void*>(&encode);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"

namespace evisel {
cudaError_t launch_probe_attn(const ProbeLaunch&, cudaStream_t) { return call("probe_attn"); }
cudaError_t launch_attn_combine(const CombineLaunch&, cudaStream_t) { return call("attn_combine"); }
cudaError_t launch_evidence(const EvidenceLaunch&, cudaStream_t) { return call("evidence"); }
cudaError_t launch_text_evidence(const TextEvidenceLaunch&, cudaStream_t) { return call("text_evidence"); }
cudaError_t launch_intra_frame(const IntraFrameLaunch&, cudaStream_t) { return call("intra_frame"); }
cudaError_t launch_cross_frame(const CrossFrameLaunch&, cudaStream_t) { return call("cross_frame"); }
cudaError_t launch_topp(const ToppLaunch&, cudaStream_t) { return call("topp"); }
cudaError_t launch_coarse(const CoarseLaunch&, cudaStream_t) { return call("coarse"); }
}  // namespace evisel
