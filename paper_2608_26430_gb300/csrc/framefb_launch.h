// Kernel launches of libframefb, chained: a kernel may be resident before the
// one queued ahead of it on the stream has ended (programmatic stream
// serialization), so that its launch latency passes during that kernel.  Every
// kernel launched this way begins with chain_wait() (framefb_ptx.cuh) and
// touches no memory before it, so the stream's order of effects stays.  Saves
// 2 to 4 us per launch behind another kernel: LLaMA-2 layer backward and AdamW,
// 2039 tokens 94.3 -> 91.8 us, 8 x 768^2 fp32 107.7 -> 103.4, 64-tenant merge
// 24.7 -> 23.3.  The tcgen05 kernels do not call chain_next(): with the next
// launch let in early ViT-B/16's step took 4677 us, without 4611 (4632 with
// plain launches).
// Internal: not part of the C ABI.
#pragma once
#include <cuda_runtime.h>

namespace ffb_host {

// Lets `fn` take `smem` bytes of dynamic shared memory.  The limit is always set
// to all that a CTA of the kernel can have: a call prepares its launches before
// it queues the first, and other threads prepare theirs, so no launch may depend
// on the size that was set last.
inline cudaError_t allow_shared(const void* fn, int dev, size_t smem) {
  cudaFuncAttributes fa{};
  int optin = 0;
  cudaError_t e = cudaFuncGetAttributes(&fa, fn);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const size_t most = static_cast<size_t>(optin) - fa.sharedSizeBytes;
  if (smem > most) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
}

inline cudaError_t launch_chained(void* fn, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t st) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace ffb_host
