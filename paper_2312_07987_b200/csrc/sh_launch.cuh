// Host-side launch helpers shared by the translation units that launch sm_100a kernels.
#pragma once
#include <mutex>
#include <utility>

#include "sh_internal.cuh"

#define SH_CUDA_CHECK(expr)                                                          \
  do {                                                                               \
    cudaError_t _e = (expr);                                                         \
    if (_e != cudaSuccess) {                                                         \
      sh_set_error("%s failed: %s", #expr, cudaGetErrorString(_e));                  \
      return SH_ERR_CUDA;                                                            \
    }                                                                                \
  } while (0)

// Kernel launch, optionally with the programmatic-stream-serialization attribute: the kernel may
// then become resident while the kernel before it in the stream is still running, and decides
// itself (griddepcontrol.wait) when it needs that kernel's results.
template <typename... P, typename... A>
static int launch_k(bool pdl, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  SH_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...));
  return SH_OK;
}

// Dynamic shared memory limit and carve-out of a kernel, set once per (kernel, device, size): the
// attributes belong to the device's copy of the function, so a process that drives several GPUs
// must set them on each.  Always the largest shared-memory carve-out: kernels of one forward pass
// share SMs (a sort block beside a GEMM CTA; the next kernel's CTAs arriving while this one
// drains), and an SM set up with a smaller carve-out has to run empty before it can be set up again.
struct SmemAttr { const void* fn; int dev; int bytes; };
static SmemAttr g_smem_attr[128];
static int g_smem_attr_n = 0;
static std::mutex g_smem_attr_mutex;     // layers may be driven from several host threads

template <typename K>
static int set_smem(K kernel, int bytes) {
  std::lock_guard<std::mutex> lock(g_smem_attr_mutex);
  int dev = 0;
  SH_CUDA_CHECK(cudaGetDevice(&dev));
  const void* fn = (const void*)kernel;
  SmemAttr* slot = nullptr;
  for (int i = 0; i < g_smem_attr_n; ++i)
    if (g_smem_attr[i].fn == fn && g_smem_attr[i].dev == dev) slot = &g_smem_attr[i];
  if (slot && slot->bytes >= bytes) return SH_OK;
  if (bytes > 48 * 1024 || !slot)
    SH_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes > 48 * 1024 ? bytes : 48 * 1024));
  if (!slot) {
    SH_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    if (g_smem_attr_n < 128) slot = &g_smem_attr[g_smem_attr_n++];
  }
  if (slot) { slot->fn = fn; slot->dev = dev; slot->bytes = bytes; }
  return SH_OK;
}
