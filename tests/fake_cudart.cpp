// The CUDA runtime calls that the library makes, without a device: copies copy
// (the "device" memory is host memory), launches and everything else only leave
// a line in a log.  Linked with the library's own object files, it lets a test
// on the CPU see what a call hands to the runtime (fake_cuda.py).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <string>

namespace {
std::string g_log;
std::map<const void *, std::string> &names() {   // host stub -> device name
  static auto *m = new std::map<const void *, std::string>;
  return *m;
}
std::map<std::pair<int, const void *>, int> g_smem;   // (device, kernel) -> dynamic limit
int g_device = 0, g_refuse = 0;
dim3 g_grid, g_block;
size_t g_shared;
void *g_stream;

template <class... A>
void line(const char *fmt, A... a) {
  char b[512];
  snprintf(b, sizeof b, fmt, a...);
  g_log += b;
}

cudaError_t launch(const void *f, dim3 grid, dim3 block, void **args, size_t smem, unsigned cluster) {
  const std::string &name = names()[f];
  const auto it = g_smem.find({g_device, f});
  if (smem > (it == g_smem.end() ? 48 * 1024 : (size_t)it->second)) return cudaErrorInvalidValue;
  line("launch %s %d %u %u %u %u %zu %u", name.c_str(), g_device, grid.x, grid.y, grid.z, block.x,
       smem, cluster);
  // arguments of the kernels whose buffers a test looks at
  const int n = name.find("k_dot_final") != std::string::npos ? 4
                : name.find("k_begin") != std::string::npos   ? 9
                : name.find("k_store_out") != std::string::npos ? 5 : 0;
  for (int i = 0; i < n; ++i) {
    unsigned long long v;
    std::memcpy(&v, args[i], 8);
    line(" %llu", v);
  }
  g_log += '\n';
  if (name.find("k_store_out") != std::string::npos) {   // the status words, which the host reads
    const void *st = *(const void **)args[3];
    void *tail = *(void **)args[4];
    if (tail) std::memcpy(tail, st, 16);
  }
  return cudaSuccess;
}

CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t rank, void *base,
                const cuuint64_t *dims, const cuuint64_t *, const cuuint32_t *box,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  line("encode %llu", (unsigned long long)base);
  for (cuuint32_t i = 0; i < rank; ++i) line(" %llu:%u", (unsigned long long)dims[i], box[i]);
  g_log += '\n';
  return CUDA_SUCCESS;
}
}  // namespace

#define FAKE extern "C" __attribute__((visibility("default")))
FAKE const char *fake_log() { return g_log.c_str(); }
FAKE void fake_clear() { g_log.clear(); }
FAKE void fake_set_device(int d) { g_device = d; }
FAKE void fake_refuse_attributes(int n) { g_refuse = n; }   // the next n times

// what compiled CUDA code registers and launches through
FAKE void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
FAKE void __cudaRegisterFatBinaryEnd(void **) {}
FAKE void __cudaUnregisterFatBinary(void **) {}
FAKE void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *,
                                 uint3 *, dim3 *, dim3 *, int *) { names()[host] = name; }
FAKE void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
FAKE unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, CUstream_st *st) {
  g_grid = g;
  g_block = b;
  g_shared = s;
  g_stream = st;
  return 0;
}
FAKE cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) {
  *g = g_grid;
  *b = g_block;
  *s = g_shared;
  std::memcpy(st, &g_stream, sizeof g_stream);
  return cudaSuccess;
}
FAKE cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
FAKE cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t s, cudaStream_t) {
  return launch((const void *)k, g, b, args, s, 1);
}

#undef cudaGetDriverEntryPoint
FAKE cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  unsigned cluster = 1;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
  return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, cluster);
}
FAKE cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (g_refuse > 0 && g_refuse--) return cudaErrorInvalidValue;
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = v;
  return cudaSuccess;
}
FAKE cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
  *n = 152 / (int)c->attrs[0].val.clusterDim.x;
  return cudaSuccess;
}
FAKE cudaError_t cudaGetDevice(int *d) {
  *d = g_device;
  return cudaSuccess;
}
FAKE cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 152;   // asked for the number of SMs only
  return cudaSuccess;
}
FAKE cudaError_t cudaGetDriverEntryPoint(const char *, void **f, unsigned long long,
                                         cudaDriverEntryPointQueryResult *q) {
  *f = (void *)encode;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
FAKE cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  std::memcpy(d, s, n);
  line("copy %d %llu %llu %zu\n", (int)k, (unsigned long long)d, (unsigned long long)s, n);
  return cudaSuccess;
}
FAKE cudaError_t cudaStreamSynchronize(cudaStream_t) {
  g_log += "sync\n";
  return cudaSuccess;
}
FAKE cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
FAKE const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
FAKE cudaError_t cudaGetLastError() { return cudaSuccess; }

// not reached by the tests' calls (no graphs, events or static scratch)
#define UNUSED(name, ...) \
  FAKE cudaError_t name(__VA_ARGS__) { return cudaErrorNotSupported; }
UNUSED(cudaGetSymbolAddress, void **, const void *)
UNUSED(cudaEventCreate, cudaEvent_t *)
UNUSED(cudaEventDestroy, cudaEvent_t)
UNUSED(cudaEventElapsedTime, float *, cudaEvent_t, cudaEvent_t)
UNUSED(cudaEventRecord, cudaEvent_t, cudaStream_t)
UNUSED(cudaEventRecordWithFlags, cudaEvent_t, cudaStream_t, unsigned)
UNUSED(cudaGraphDestroy, cudaGraph_t)
UNUSED(cudaGraphExecDestroy, cudaGraphExec_t)
UNUSED(cudaGraphInstantiate, cudaGraphExec_t *, cudaGraph_t, unsigned long long)
UNUSED(cudaGraphLaunch, cudaGraphExec_t, cudaStream_t)
UNUSED(cudaStreamBeginCapture, cudaStream_t, cudaStreamCaptureMode)
UNUSED(cudaStreamCreateWithFlags, cudaStream_t *, unsigned)
UNUSED(cudaStreamDestroy, cudaStream_t)
UNUSED(cudaStreamEndCapture, cudaStream_t, cudaGraph_t *)
