// A CUDA runtime of fake devices for tests of the library's host side: linked
// with the library's objects in place of the CUDA runtime.  Two devices of
// compute capability 10.3 with 152 SMs; "device memory" is host memory; no
// kernel runs, but launches are checked as a device checks them (dynamic
// shared memory above 48 KB and clusters above 8 need the kernel's attribute
// on the device that is current), and the kernels that count spikes have the
// effect of their count.
#include <cuda.h>
#include <cuda_runtime.h>

#include <chrono>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <thread>
#include <utility>
#include <vector>

#include "sp_internal.h"

namespace {

constexpr int kDevices = 2;
struct State {
  int device = 0;
  std::map<const void*, std::string> kernels;                  // host stub -> name
  std::map<std::pair<int, const void*>, int> smem, nonportable;   // (device, kernel) -> attribute
  std::string fail;                                            // launches of kernels with this in the name fail
  int active = 0;                                              // spikes that a counting kernel finds
  int publish_ms = 0;                                          // delay of a publication (< 0: it never comes)
  std::string last;                                            // the kernel launched last
  int launches = 0, synced = -1;                               // synced: the device last synchronised
  size_t pushed_smem = 0;                                      // of a <<<...>>> launch
  std::vector<std::thread> pending;
};
State& state() {
  static State s;
  return s;
}

void finish_pending() {
  for (auto& t : state().pending) t.join();
  state().pending.clear();
}

void publish(const sp::SpikeCount& c) {
  const uint32_t count = (uint32_t)c.dev[0];
  c.dev[0] = c.dev[1] = 0;
  const int ms = state().publish_ms;
  if (ms < 0) return;
  const auto store = [c, count] {
    __atomic_store_n(c.host, (uint64_t)c.seq << 32 | count, __ATOMIC_RELEASE);
  };
  if (ms == 0) return store();
  state().pending.emplace_back([store, ms] {
    std::this_thread::sleep_for(std::chrono::milliseconds(ms));
    store();
  });
}

cudaError_t launch(const void* f, size_t smem, unsigned cluster, void** args) {
  State& s = state();
  const std::string& name = s.kernels.at(f);
  const std::pair<int, const void*> key{s.device, f};
  if (!s.fail.empty() && name.find(s.fail) != std::string::npos) return cudaErrorLaunchOutOfResources;
  if (smem > 48 * 1024 && s.smem[key] < (int)smem) return cudaErrorInvalidValue;
  if (cluster > 8 && !s.nonportable[key]) return cudaErrorInvalidClusterSize;
  ++s.launches;
  s.last = name;
  if (name.find("spikes_to_01_kernel") != std::string::npos) {
    const auto& c = *static_cast<const sp::SpikeCount*>(args[7]);
    if (c.dev) c.dev[0] += s.active;
  } else if (name.find("density_kernel") != std::string::npos) {
    const auto& c = *static_cast<const sp::SpikeCount*>(args[5]);
    c.dev[0] += s.active;
    publish(c);
  } else if (name.find("gemm_kernel") != std::string::npos) {
    const auto& p = *static_cast<const sp::GemmParams*>(args[2]);
    if (p.count.dev) publish(p.count);
  }
  return cudaSuccess;
}

CUresult encode_tiled(CUtensorMap*, ...) { return CUDA_SUCCESS; }

}  // namespace

extern "C" {

// ---- test controls ----------------------------------------------------------
void fake_fail(const char* name) { state().fail = name; }
void fake_counts(int active, int publish_ms) {
  state().active = active;
  state().publish_ms = publish_ms;
}
void fake_device(int device) { state().device = device; }
int fake_launches() { return std::exchange(state().launches, 0); }
int fake_last_is(const char* name) { return state().last.find(name) != std::string::npos; }
int fake_synced() { return std::exchange(state().synced, -1); }

// ---- the runtime ------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&state()); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
  state().kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, struct CUstream_st*) {
  state().pushed_smem = smem;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void*) {
  *smem = state().pushed_smem;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* kernel, const void* f) {
  *kernel = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void** args, size_t smem, cudaStream_t) {
  return launch(kernel, smem, 1, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void** args) {
  unsigned cluster = 1;
  for (unsigned i = 0; i < cfg->numAttrs; ++i)
    if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = cfg->attrs[i].val.clusterDim.x;
  return launch(f, cfg->dynamicSmemBytes, cluster, args);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute attr, int value) {
  const std::pair<int, const void*> key{state().device, f};
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) state().smem[key] = value;
  if (attr == cudaFuncAttributeNonPortableClusterSizeAllowed) state().nonportable[key] = value;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* device) {
  *device = state().device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int device) {
  if (device < 0 || device >= kDevices) return cudaErrorInvalidDevice;
  state().device = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr attr, int) {
  *value = attr == cudaDevAttrComputeCapabilityMajor ? 10
           : attr == cudaDevAttrComputeCapabilityMinor ? 3
           : attr == cudaDevAttrMultiProcessorCount ? 152
                                                    : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
  state().synced = state().device;
  finish_pending();
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  finish_pending();
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* status) {
  *status = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemsetAsync(void* p, int value, size_t n, cudaStream_t) {
  std::memset(p, value, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  *p = const_cast<void*>(symbol);
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* result) {
  *fn = reinterpret_cast<void*>(encode_tiled);
  *result = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* cfg) {
  const State& s = state();
  const auto it = s.smem.find({s.device, f});
  if (cfg->dynamicSmemBytes > 48 * 1024 && (it == s.smem.end() || it->second < (int)cfg->dynamicSmemBytes))
    return cudaErrorInvalidValue;
  *n = 152 / (int)cfg->attrs[0].val.clusterDim.x;
  return cudaSuccess;
}

}  // extern "C"
