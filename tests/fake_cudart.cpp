// A stand-in for the CUDA runtime, linked with the library's own object files
// in the place of libcudart: the host code (plans, dispatch, per-device state,
// error paths) then runs without a GPU.  No kernel runs; launches are checked
// against the attributes set on the current device and recorded.  Device
// memory is host memory, graphs record nothing, and event times come from
// costs that a test gives per kernel.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Launch {
  int device;
  std::string name;
  unsigned grid, block, cluster;
  size_t smem;
};
struct Cost {
  std::string name;
  double us, first;
  int arg;  // >= 0: `us` is per unit of this int argument
};

int g_device = 0;
std::map<const void *, std::string> g_names;
std::map<std::pair<int, const void *>, std::map<int, int>> g_attr;  // (device, kernel) -> attribute -> value
std::map<const void *, int> g_launched;
std::vector<Launch> g_log;
std::vector<Cost> g_costs;
std::map<cudaEvent_t, double> g_events;
double g_now = 0.0;       // us
std::string g_watch;      // kernel whose argument g_watch_arg is copied at each launch
int g_watch_arg = 0;
std::vector<char> g_watched;
int g_clusters = 9;       // clusters that the device holds at once
int g_fail_clusters = 0;  // cluster queries to fail
int g_fail_malloc = 0;    // the allocation to fail, counted from now (0: none)
dim3 g_grid, g_block;
size_t g_smem;
cudaStream_t g_stream;

int attr(const void *f, int a) { return g_attr[{g_device, f}][a]; }

cudaError_t record(const void *f, dim3 grid, dim3 block, size_t smem, unsigned cluster, void **args) {
  if (smem > 48 * 1024 && (size_t)attr(f, cudaFuncAttributeMaxDynamicSharedMemorySize) < smem)
    return cudaErrorInvalidValue;
  if (cluster > 8 && !attr(f, cudaFuncAttributeNonPortableClusterSizeAllowed)) return cudaErrorInvalidClusterSize;
  if (!grid.x || !grid.y || !grid.z || !block.x) return cudaErrorInvalidConfiguration;
  g_log.push_back({g_device, g_names[f], grid.x * grid.y * grid.z, block.x, cluster, smem});
  for (const Cost &c : g_costs)
    if (g_names[f].find(c.name) != std::string::npos) {
      g_now += c.us * (c.arg < 0 ? 1 : *static_cast<int *>(args[c.arg])) + (g_launched[f] ? 0.0 : c.first);
      break;
    }
  ++g_launched[f];
  if (!g_watch.empty() && g_names[f].find(g_watch) != std::string::npos)
    std::memcpy(g_watched.data(), args[g_watch_arg], g_watched.size());
  return cudaSuccess;
}

cudaError_t allocate(void **p, size_t n) {
  if (g_fail_malloc && --g_fail_malloc == 0) return cudaErrorMemoryAllocation;
  *p = std::calloc(n ? n : 1, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}

CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- what the tests set and read
void fake_reset() {
  g_log.clear();
  g_costs.clear();
  g_launched.clear();
  g_watch.clear();
  g_clusters = 9;
  g_fail_clusters = g_fail_malloc = 0;
}
void fake_set_device(int d) { g_device = d; }
void fake_clusters(int n) { g_clusters = n; }
void fake_fail_clusters(int n) { g_fail_clusters = n; }
void fake_fail_malloc(int n) { g_fail_malloc = n; }
void fake_cost(const char *name, double us, double first, int arg) { g_costs.push_back({name, us, first, arg}); }
void fake_watch(const char *name, int arg, int bytes) {
  g_watch = name;
  g_watch_arg = arg;
  g_watched.assign(bytes, 0);
}
const char *fake_watched() { return g_watched.data(); }
void fake_clear() { g_log.clear(); }
int fake_launches() { return (int)g_log.size(); }
const char *fake_launch(int k, int *device, unsigned *grid, unsigned *block, unsigned *cluster) {
  const Launch &l = g_log[k];
  *device = l.device;
  *grid = l.grid;
  *block = l.block;
  *cluster = l.cluster;
  return l.name.c_str();
}

// ---- the runtime
void **__cudaRegisterFatBinary(void *) {
  static void *handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, CUstream_st *s) {
  g_grid = grid;
  g_block = block;
  g_smem = smem;
  g_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
  *grid = g_grid;
  *block = g_block;
  *smem = g_smem;
  *static_cast<cudaStream_t *>(s) = g_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
  return cudaSuccess;
}
static cudaError_t g_last = cudaSuccess;
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t) {
  const cudaError_t e = record(k, grid, block, smem, 1, args);
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  unsigned cluster = 1;
  for (unsigned k = 0; k < c->numAttrs; ++k)
    if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[k].val.clusterDim.x;
  const cudaError_t e = record(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster, args);
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "stand-in error"; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  g_attr[{g_device, f}][a] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
  unsigned cluster = 1;
  for (unsigned k = 0; k < c->numAttrs; ++k)
    if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[k].val.clusterDim.x;
  cudaError_t e = cudaSuccess;
  if (g_fail_clusters > 0) {
    --g_fail_clusters;
    e = cudaErrorUnknown;
  } else if (c->dynamicSmemBytes > 48 * 1024 &&
             (size_t)attr(f, cudaFuncAttributeMaxDynamicSharedMemorySize) < c->dynamicSmemBytes) {
    e = cudaErrorInvalidValue;
  } else if (cluster > 8 && !attr(f, cudaFuncAttributeNonPortableClusterSizeAllowed)) {
    e = cudaErrorInvalidClusterSize;
  }
  if (e != cudaSuccess) g_last = e;
  else *n = g_clusters;
  return e;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int block, size_t smem,
                                                                   unsigned) {
  *n = (int)std::min<size_t>({2048u / (unsigned)block, 8, 228 * 1024 / (smem + 1024)});
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  g_device = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 152;  // asked for the number of SMs only
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return allocate(p, n); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return allocate(p, n); }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return std::free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = reinterpret_cast<cudaEvent_t>(std::malloc(1));
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return g_events[e] = g_now, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)((g_events[b] - g_events[a]) / 1e3);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(std::malloc(1));
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  *a = cudaPointerAttributes{};
  a->device = g_device;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return *p = nullptr, cudaErrorInvalidSymbol; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *p = reinterpret_cast<void *>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
