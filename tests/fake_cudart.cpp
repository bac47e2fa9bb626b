// A stand-in for the CUDA runtime with two devices and no GPU: linked with the library's objects in
// place of libcudart, it lets a test follow what the host code asks of the runtime. Device memory is
// host memory, kernels do not run. What it holds to is what a device would refuse: a launch with more
// dynamic shared memory than the kernel was opted into ON THAT DEVICE, and the pending last error.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <utility>
#include <vector>

#define EXPORT extern "C" __attribute__((visibility("default")))

namespace {
constexpr int kDefaultSmem = 48 * 1024;
int g_device = 0, g_skip = 0, g_fail = 0;  // the next launches to let through, then to fail
cudaError_t g_last = cudaSuccess;
std::map<std::pair<int, const void*>, int> g_smem;  // (device, kernel) -> opted-in bytes
struct Launch { std::string kernel; int early, watched; };  // early: with programmatic serialisation
std::vector<Launch> g_launches;
std::map<const void*, std::string> g_names;
int g_watch = -1;  // byte offset of an int in the first argument of the kernels, kept with each launch
struct Call { dim3 grid, block; size_t smem; void* stream; };
std::vector<Call> g_calls;

cudaError_t ret(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t launch(const void* f, size_t smem, int early, void** args) {
  if (g_skip > 0) {
    --g_skip;
  } else if (g_fail > 0) {
    --g_fail;
    return ret(cudaErrorLaunchOutOfResources);
  }
  auto it = g_smem.find({g_device, f});
  if ((long long)smem > (it == g_smem.end() ? kDefaultSmem : it->second)) return ret(cudaErrorInvalidValue);
  int watched = 0;
  if (g_watch >= 0) memcpy(&watched, (const char*)args[0] + g_watch, sizeof(int));
  g_launches.push_back({g_names[f], early, watched});
  return cudaSuccess;
}
CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
}  // namespace

// ---- the test's side
EXPORT void fake_fail_launches(int skip, int n) { g_skip = skip; g_fail = n; }
EXPORT int fake_launches() { return (int)g_launches.size(); }
EXPORT const char* fake_launch_kernel(int i) { return g_launches[i].kernel.c_str(); }
EXPORT void fake_watch(int offset) { g_watch = offset; }
EXPORT int fake_watched(int i) { return g_launches[i].watched; }
EXPORT int fake_launch_early(int i) { return g_launches[i].early; }
EXPORT int fake_last_error() { return (int)g_last; }
EXPORT int fake_set_device(int d) { return cudaSetDevice(d); }

// ---- the runtime's side
EXPORT void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
EXPORT void __cudaRegisterFatBinaryEnd(void**) {}
EXPORT void __cudaUnregisterFatBinary(void**) {}
EXPORT void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
EXPORT void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[f] = name;
}
EXPORT unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  g_calls.push_back({g, b, smem, s});
  return 0;
}
EXPORT cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  const Call c = g_calls.back();
  g_calls.pop_back();
  *g = c.grid;
  *b = c.block;
  *smem = c.smem;
  *(void**)s = c.stream;
  return cudaSuccess;
}
EXPORT cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
EXPORT cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t smem, cudaStream_t) {
  return launch((const void*)k, smem, 0, args);
}
EXPORT cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  int early = 0;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    early |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
             c->attrs[i].val.programmaticStreamSerializationAllowed;
  return launch(f, c->dynamicSmemBytes, early, args);
}
EXPORT cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = v;
  return cudaSuccess;
}
EXPORT cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
EXPORT cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
EXPORT cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d > 1) return ret(cudaErrorInvalidDevice);
  g_device = d;
  return cudaSuccess;
}
EXPORT cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
EXPORT cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
EXPORT const char* cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }
EXPORT cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                                    cudaDriverEntryPointQueryResult* q) {
  *p = (void*)&encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
EXPORT cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char scratch[1 << 16];
  *p = scratch;
  return cudaSuccess;
}
EXPORT cudaError_t cudaMalloc(void** p, size_t n) { *p = aligned_alloc(512, (n + 511) / 512 * 512); return *p ? cudaSuccess : ret(cudaErrorMemoryAllocation); }
EXPORT cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
EXPORT cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
EXPORT cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
EXPORT cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
EXPORT cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)8; return cudaSuccess; }
EXPORT cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
EXPORT cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
EXPORT cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
EXPORT cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) { *st = cudaStreamCaptureStatusNone; return cudaSuccess; }
EXPORT cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
EXPORT cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)8; return cudaSuccess; }
EXPORT cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)8; return cudaSuccess; }
EXPORT cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)8; return cudaSuccess; }
EXPORT cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
EXPORT cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
EXPORT cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
EXPORT cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
EXPORT cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
EXPORT cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
EXPORT cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) { return cudaSuccess; }
EXPORT cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)8; return cudaSuccess; }
EXPORT cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
