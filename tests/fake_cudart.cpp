// A CUDA runtime without a device: the library's objects link against it instead of cudart, so that its host code
// (checks, routes, launch configurations, what it keeps per device) runs and is recorded on a machine without a GPU.
// "Device" memory is host memory, or addresses from 2^44 on that hold nothing; kernels do nothing.  A launch is refused as the driver refuses it where the current
// device's kernel attributes do not allow its shared memory or its cluster.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <cxxabi.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Launch {
  std::string kernel;
  int device, grid, block, cluster, cooperative, arg;
  size_t smem;
};
struct Attrs {
  size_t smem = 48 * 1024;
  bool wide = false;
};

std::mutex mu;
std::map<const void*, std::string> kernels;
std::map<std::pair<int, const void*>, Attrs> attrs;
std::map<std::pair<int, const void*>, void*> symbols;
std::vector<Launch> launches;
std::vector<int> boxes;              // rows of the tensor maps' boxes
std::map<std::string, int> wanted;   // part of a kernel's name -> the int argument to record
thread_local int device = 0;
thread_local struct {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} pushed;
const int sms = 152;

// Clusters of one-CTA-per-SM kernels that are resident at once: a cluster stays in a group of SMs (76 of two CTAs, 36 of
// four, 15 of eight and 7 of sixteen, as a GB300 answers).
int clusters(int size) {
  int n = 0;
  for (int group : {18, 18, 20, 20, 20, 20, 22, 14}) n += group / size;
  return n;
}

cudaError_t launch(const void* func, dim3 grid, dim3 block, size_t smem, int cluster, int cooperative, void** args) {
  std::lock_guard<std::mutex> lock(mu);
  const Attrs a = attrs[{device, func}];
  if (smem > a.smem) return cudaErrorInvalidValue;
  if (cluster > 8 && !a.wide) return cudaErrorInvalidClusterSize;
  if (grid.x % cluster) return cudaErrorInvalidValue;
  if (cooperative && (int)(grid.x * grid.y * grid.z) > sms) return cudaErrorCooperativeLaunchTooLarge;
  Launch l{kernels[func], device, (int)(grid.x * grid.y * grid.z), (int)block.x, cluster, cooperative, -1, smem};
  for (const auto& w : wanted)
    if (l.kernel.find(w.first) != std::string::npos) std::memcpy(&l.arg, args[w.second], sizeof(int));
  launches.push_back(l);
  return cudaSuccess;
}

bool backed(const void* p) { return (uintptr_t)p >> 40 != 0x10; }

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t* box, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
  boxes.push_back((int)box[1]);
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- what a test asks -------------------------------------------------------------------------
void fake_reset() {
  std::lock_guard<std::mutex> lock(mu);
  launches.clear();
  boxes.clear();
}
void fake_set_device(int d) { device = d; }
void fake_record_arg(const char* kernel, int index) { wanted[kernel] = index; }
int fake_boxes() { return (int)boxes.size(); }
int fake_box_rows(int i) { return boxes[i]; }
int fake_launches() { return (int)launches.size(); }
const char* fake_kernel(int i) { return launches[i].kernel.c_str(); }
int fake_field(int i, int which) {
  const Launch& l = launches[i];
  const int f[] = {l.device, l.grid, l.block, l.cluster, l.cooperative, l.arg, (int)l.smem};
  return f[which];
}

// ---- the runtime ------------------------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) {
  static void* handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  int status = 0;
  char* text = abi::__cxa_demangle(name, nullptr, nullptr, &status);
  kernels[host] = status == 0 ? text : name;
  std::free(text);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* stream) {
  pushed = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = pushed.grid;
  *block = pushed.block;
  *smem = pushed.smem;
  *static_cast<cudaStream_t*>(stream) = pushed.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* kernel, const void* host) {
  *kernel = (cudaKernel_t)host;
  return cudaSuccess;
}
thread_local cudaError_t last = cudaSuccess;
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t) {
  const cudaError_t e = launch((const void*)kernel, grid, block, smem, 1, 0, args);
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void** args) {
  int cluster = 1, cooperative = 0;
  for (unsigned i = 0; i < c->numAttrs; ++i) {
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = (int)c->attrs[i].val.clusterDim.x;
    if (c->attrs[i].id == cudaLaunchAttributeCooperative) cooperative = c->attrs[i].val.cooperative;
  }
  return launch(func, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster, cooperative, args);
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "refused by the fake runtime"; }
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrComputeCapabilityMajor ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3 : a == cudaDevAttrCooperativeLaunch ? 1 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* func, enum cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> lock(mu);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) attrs[{device, func}].smem = (size_t)v;
  if (a == cudaFuncAttributeNonPortableClusterSizeAllowed) attrs[{device, func}].wide = v != 0;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* func, const cudaLaunchConfig_t* c) {
  std::lock_guard<std::mutex> lock(mu);
  int size = 2;                                       // kernels with __cluster_dims__ are pairs
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) size = (int)c->attrs[i].val.clusterDim.x;
  if (size > 8 && !attrs[{device, func}].wide) return cudaErrorInvalidClusterSize;
  *n = clusters(size);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             enum cudaDriverEntryPointQueryResult* q) {
  *fn = (void*)encode;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  std::lock_guard<std::mutex> lock(mu);
  void*& at = symbols[{device, symbol}];
  if (!at) at = std::calloc(1, 16 << 20);
  *p = at;
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) {
  *p = std::calloc(1, bytes);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t bytes, enum cudaMemcpyKind, cudaStream_t) {
  if (backed(dst) && backed(src)) std::memcpy(dst, src, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) {
  if (backed(p)) std::memset(p, v, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbol(void* dst, const void*, size_t bytes, size_t, enum cudaMemcpyKind) {
  std::memset(dst, 0, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, enum cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }

}  // extern "C"
