// Run-time compilation of the generated fused / batched kernels for sm_103a.
//
// Compilation (NVRTC, source -> CUBIN) needs no GPU; loading (cudaLibraryLoadData)
// does.  Compiled kernels are cached for the life of the process, keyed by their full
// source text, so plans with the same program share one kernel.
#include <cuda_runtime.h>
#include <nvrtc.h>

#include <algorithm>
#include <memory>
#include <mutex>
#include <string>
#include <unordered_map>

#include "gar_internal.hpp"

namespace gar {
namespace {

// never destroyed: a plan may be destroyed after this file's static objects would be
std::mutex &g_mu = *new std::mutex;
std::unordered_map<std::string, std::unique_ptr<JitKernel>> &g_cache =
    *new std::unordered_map<std::string, std::unique_ptr<JitKernel>>;

}  // namespace

int jit_compile(const CodegenResult &cg, JitKernel **out) {
  std::lock_guard<std::mutex> lock(g_mu);
  auto it = g_cache.find(cg.source);
  if (it != g_cache.end()) {
    *out = it->second.get();
    return GAR_OK;
  }
  nvrtcProgram prog;
  if (nvrtcCreateProgram(&prog, cg.source.c_str(), "gar_generated.cu", 0, nullptr, nullptr) !=
      NVRTC_SUCCESS) {
    set_error("nvrtcCreateProgram failed");
    return GAR_EJIT;
  }
  const char *opts[] = {"--gpu-architecture=sm_103a", "--std=c++17", "-lineinfo",
                        "--fmad=false", "--ftz=false", "--prec-div=true", "--prec-sqrt=true"};
  nvrtcResult rc = nvrtcCompileProgram(prog, (int)(sizeof opts / sizeof opts[0]), opts);
  if (rc != NVRTC_SUCCESS) {
    size_t n = 0;
    nvrtcGetProgramLogSize(prog, &n);
    std::string log(n, '\0');
    if (n) nvrtcGetProgramLog(prog, &log[0]);
    nvrtcDestroyProgram(&prog);
    set_error("NVRTC compile of " + cg.kernel_name + " failed: " + log);
    return GAR_EJIT;
  }
  size_t bytes = 0;
  if (nvrtcGetCUBINSize(prog, &bytes) != NVRTC_SUCCESS || bytes == 0) {
    nvrtcDestroyProgram(&prog);
    set_error("NVRTC produced no CUBIN for " + cg.kernel_name);
    return GAR_EJIT;
  }
  auto k = std::make_unique<JitKernel>();
  k->cubin.resize(bytes);
  nvrtcGetCUBIN(prog, k->cubin.data());
  nvrtcDestroyProgram(&prog);
  k->name = cg.kernel_name;
  k->source = cg.source;
  k->width = cg.width;
  k->host_width = cg.host_width;
  k->table_copies = cg.table_copies;
  k->threads = cg.threads;
  k->form = cg.form;
  k->smem = cg.smem;
  k->tile = cg.tile;
  *out = k.get();
  g_cache.emplace(cg.source, std::move(k));
  return GAR_OK;
}

namespace {

int load_library(JitKernel *k) {
  cudaLibrary_t lib = nullptr;
  cudaError_t e = cudaLibraryLoadData(&lib, k->cubin.data(), nullptr, nullptr, 0, nullptr,
                                      nullptr, 0);
  if (e != cudaSuccess) return cuda_fail(e, "cudaLibraryLoadData");
  cudaKernel_t kern = nullptr;
  e = cudaLibraryGetKernel(&kern, lib, k->name.c_str());
  if (e != cudaSuccess) {
    cudaLibraryUnload(lib);
    return cuda_fail(e, "cudaLibraryGetKernel");
  }
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, (const void *)kern) == cudaSuccess) {
    k->regs = fa.numRegs;
    k->local_bytes = (int)fa.localSizeBytes;
  } else {
    cudaGetLastError();
  }
  k->library = lib;
  k->kernel = (void *)kern;
  k->loaded = true;
  return GAR_OK;
}

}  // namespace

// The library and its kernel serve every device; the shared-memory limit, the resident CTAs
// and the addresses of the kernel's variables are a device's own.
int jit_load(JitKernel *k, JitOnDevice *here) {
  std::lock_guard<std::mutex> lock(g_mu);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (!k->loaded)
    if (int rc = load_library(k)) return rc;
  if (k->on.size() <= (size_t)dev) k->on.resize((size_t)dev + 1);
  JitOnDevice &on = k->on[(size_t)dev];
  if (on.blocks_per_sm == 0) {
    if (k->smem > 32 * 1024) {  // (and the kernel's static shared memory)
      e = cudaFuncSetAttribute((const void *)k->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, k->smem);
      if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(dynamic shared memory)");
    }
    if (k->form == GAR_FORM_STREAM) {
      size_t bytes = 0;
      e = cudaLibraryGetGlobal(&on.gave_up, &bytes, (cudaLibrary_t)k->library, "gar_gave_up");
      if (e != cudaSuccess) return cuda_fail(e, "cudaLibraryGetGlobal");
    }
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void *)k->kernel, k->threads, k->smem);
    if (e != cudaSuccess || nb <= 0) {
      cudaGetLastError();
      nb = 1;
    }
    on.blocks_per_sm = nb;
  }
  if (here != nullptr) *here = on;
  return GAR_OK;
}

int jit_take_slot(JitKernel *k, int dev, unsigned int *seen) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (k->slots.size() <= (size_t)dev) k->slots.resize((size_t)dev + 1);
  WaitSlots &w = k->slots[(size_t)dev];
  const int slot = (int)(std::min_element(w.users, w.users + GAR_WAIT_SLOTS) - w.users);
  ++w.users[slot];
  *seen = w.seen[slot];
  return slot;
}

void jit_seen_slot(JitKernel *k, int dev, int slot, unsigned int seen) {
  std::lock_guard<std::mutex> lock(g_mu);
  k->slots[(size_t)dev].seen[slot] = seen;
}

void jit_drop_slot(JitKernel *k, int dev, int slot) {
  std::lock_guard<std::mutex> lock(g_mu);
  --k->slots[(size_t)dev].users[slot];
}

}  // namespace gar
