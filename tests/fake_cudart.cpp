// A stand-in for the CUDA runtime, linked with the library's objects in place of the real one, so
// that the host code that chooses kernels runs without a GPU: launches are recorded by kernel name
// and grid, and a test sets what the device queries answer.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>
#include <map>
#include <string>

namespace {
std::map<const void*, std::string> g_names;
std::string g_log;
int g_device, g_sms = 152, g_clusters[2] = {76, 36}, g_cluster_error, g_cluster_queries;
char g_symbol[256];

// a kernel's flag on the order of dependent launches: lora_down's `settle`, the GEMV's `x_settled`
int order_flag(const std::string& name, void** args) {
  if (name.find("lora_down") != std::string::npos) return *static_cast<int*>(args[8]);
  if (name.find("dual_lora_gemv") != std::string::npos) return *static_cast<int*>(args[13]);
  return -1;
}

void record(const void* fn, dim3 grid, unsigned cluster, void** args) {
  auto it = g_names.find(fn);
  const std::string name = it == g_names.end() ? "?" : it->second;
  g_log += name + " " + std::to_string(grid.x) + " " + std::to_string(grid.y) + " " + std::to_string(grid.z) + " " +
           std::to_string(cluster) + " " + std::to_string(order_flag(name, args)) + "\n";
}

CUresult encode_tiled(CUtensorMap* map, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                      const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  std::memset(map, 0, sizeof *map);
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {

// what the test sets and reads
void fake_device(int device, int sms, int pair_clusters, int quad_clusters, int cluster_error) {
  g_device = device;
  g_sms = sms;
  g_clusters[0] = pair_clusters;
  g_clusters[1] = quad_clusters;
  g_cluster_error = cluster_error;
}
int fake_cluster_queries() { return g_cluster_queries; }
const char* fake_launches() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
const char* fake_kernels() {  // every kernel of the library, one per line
  static std::string all;
  all.clear();
  for (auto& n : g_names) all += n.second + "\n";
  return all.c_str();
}

// the runtime's functions that the library calls
cudaError_t cudaGetDevice(int* d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = g_sms, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = g_symbol, cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void* dst, const void*, size_t n, size_t, cudaMemcpyKind) {
  return std::memset(dst, 0, n), cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 4, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* cfg) {
  ++g_cluster_queries;
  if (g_cluster_error) return cudaErrorUnknown;
  return *n = g_clusters[cfg->attrs[0].val.clusterDim.x > 2], cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(&encode_tiled);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* fn, void** args) {
  unsigned cluster = 1;
  for (unsigned i = 0; i < cfg->numAttrs; ++i)
    if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = cfg->attrs[i].val.clusterDim.x;
  return record(fn, cfg->gridDim, cluster, args), cudaSuccess;
}

// what the compiler's registration and launch stubs call
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void*) {
  return *grid = dim3(), *block = dim3(), *smem = 0, cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
  return *k = static_cast<cudaKernel_t>(const_cast<void*>(fn)), cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t, cudaStream_t) {
  return record(k, grid, 1, args), cudaSuccess;
}
}
