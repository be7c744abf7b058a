// A CUDA runtime and NVRTC in plain C++ for host tests of the library's host code: several
// devices, memory and streams that are the host's own, kernels that are recorded and not
// run.  Linked in place of libcudart and libnvrtc.
#pragma once

#include <cuda_runtime.h>
#include <nvrtc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "gar.h"
#include "gar_internal.hpp"

#define CHECK(cond)                                                                  \
  do {                                                                               \
    if (!(cond)) {                                                                   \
      std::printf("%s:%d: %s (%s)\n", __FILE__, __LINE__, #cond, gar_last_error());  \
      std::exit(1);                                                                  \
    }                                                                                \
  } while (0)

namespace fake {

struct Launch {
  std::string kernel;
  int device;
  unsigned grid, block;
  size_t smem;
  cudaStream_t stream;
  void **args;
};

struct Function {
  std::string source, name;
  std::map<int, int> smem_limit;                               // by device
  std::map<std::pair<int, std::string>, std::vector<char>> globals;  // by device and name
};

inline std::mutex mu;
inline thread_local int device = 0;
inline std::map<int, int> sms = {{0, 152}, {1, 152}};
inline std::function<int(int)> blocks_per_sm = [](int) { return 1; };
inline int local_bytes = 0, regs = 64;
inline int compiles = 0;
inline std::vector<Launch> launches;
inline std::function<cudaError_t(Function &, const Launch &)> on_launch;
inline std::function<cudaError_t(cudaStream_t)> on_synchronize;
inline cudaMemoryType memory = cudaMemoryTypeDevice;
inline std::string last_source;
inline cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;

}  // namespace fake

struct _nvrtcProgram {
  std::string source;
};

extern "C" {

nvrtcResult nvrtcCreateProgram(nvrtcProgram *p, const char *src, const char *, int, const char *const *, const char *const *) {
  *p = new _nvrtcProgram{src};
  return NVRTC_SUCCESS;
}
nvrtcResult nvrtcCompileProgram(nvrtcProgram, int, const char *const *) {
  std::lock_guard<std::mutex> lock(fake::mu);
  ++fake::compiles;
  return NVRTC_SUCCESS;
}
nvrtcResult nvrtcDestroyProgram(nvrtcProgram *p) {
  delete *p;
  return NVRTC_SUCCESS;
}
nvrtcResult nvrtcGetProgramLogSize(nvrtcProgram, size_t *n) { return *n = 0, NVRTC_SUCCESS; }
nvrtcResult nvrtcGetProgramLog(nvrtcProgram, char *) { return NVRTC_SUCCESS; }
nvrtcResult nvrtcGetCUBINSize(nvrtcProgram p, size_t *n) { return *n = p->source.size() + 1, NVRTC_SUCCESS; }
nvrtcResult nvrtcGetCUBIN(nvrtcProgram p, char *out) { return std::memcpy(out, p->source.c_str(), p->source.size() + 1), NVRTC_SUCCESS; }

cudaError_t cudaGetDevice(int *d) { return *d = fake::device, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int d) {
  return *v = a == cudaDevAttrMultiProcessorCount ? fake::sms[d] : 0, cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { return *p = std::aligned_alloc(256, (n + 255) / 256 * 256), cudaSuccess; }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = (cudaStream_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free((void *)s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return fake::on_synchronize ? fake::on_synchronize(s) : cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) { return *st = fake::capture, cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = (cudaEvent_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free((void *)e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  *a = cudaPointerAttributes{};
  a->type = fake::memory;
  a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}

cudaError_t cudaLibraryLoadData(cudaLibrary_t *lib, const void *code, cudaJitOption *, void **, unsigned, cudaLibraryOption *,
                                void **, unsigned) {
  auto *f = new fake::Function;
  f->source = static_cast<const char *>(code);
  *lib = reinterpret_cast<cudaLibrary_t>(f);
  return cudaSuccess;
}
cudaError_t cudaLibraryUnload(cudaLibrary_t lib) { return delete reinterpret_cast<fake::Function *>(lib), cudaSuccess; }
cudaError_t cudaLibraryGetKernel(cudaKernel_t *k, cudaLibrary_t lib, const char *name) {
  reinterpret_cast<fake::Function *>(lib)->name = name;
  *k = reinterpret_cast<cudaKernel_t>(lib);
  return cudaSuccess;
}
cudaError_t cudaLibraryGetGlobal(void **p, size_t *bytes, cudaLibrary_t lib, const char *name) {
  auto *f = reinterpret_cast<fake::Function *>(lib);
  if (f->source.find(name) == std::string::npos) return cudaErrorSymbolNotFound;
  auto &v = f->globals[{fake::device, name}];
  if (v.empty()) v.resize(4096);
  *p = v.data();
  *bytes = v.size();
  return cudaSuccess;
}
// The attribute belongs to the current device, as CUDA's does.
cudaError_t cudaFuncSetAttribute(const void *k, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) ((fake::Function *)k)->smem_limit[fake::device] = v;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  *a = cudaFuncAttributes{};
  a->numRegs = fake::regs;
  a->localSizeBytes = (size_t)fake::local_bytes;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
  return *n = fake::blocks_per_sm(fake::device), cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *k, void **args) {
  auto &f = *(fake::Function *)k;
  const size_t smem = cfg->dynamicSmemBytes;
  std::lock_guard<std::mutex> lock(fake::mu);
  if (smem > 48 * 1024 && (size_t)f.smem_limit[fake::device] < smem) return cudaErrorInvalidValue;
  fake::launches.push_back({f.name, fake::device, cfg->gridDim.x, cfg->blockDim.x, smem, cfg->stream, args});
  return fake::on_launch ? fake::on_launch(f, fake::launches.back()) : cudaSuccess;
}

}  // extern "C"

// The step kernels' host side, which the checks do not use.
namespace gar {
int num_sms() { return fake::sms[fake::device]; }
int launch_step(const gar_plan &, const Launch &, int, void *const *, gar_stream_t) { return GAR_EINVAL; }
int launch_persistent(const gar_plan &, void *const *, gar_stream_t) { return GAR_EINVAL; }
size_t barrier_state_bytes() { return 64; }
void barrier_outcome(const void *, int *error, int *launch) { *error = *launch = 0; }
LaunchDesc launch_desc(const gar_plan &, const Launch &) { return {}; }
int load_step_module() { return GAR_OK; }
}  // namespace gar
