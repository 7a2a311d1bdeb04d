// Launch helper: programmatic dependent launch.
#pragma once

#include <cuda_runtime.h>

namespace alr {

// Launch attribute of the library's kernels: a kernel may be scheduled while the kernel before it
// in the stream is still running, sets itself up (barriers, tensor memory, tensor-map fetches),
// waits (pdl_wait in the kernel, before any global access) until that kernel has completed and its
// writes are visible, and lets the kernel after it be scheduled early in turn (pdl_release).
// Every thread of every kernel waits, so a kernel's completion implies that of all before it in
// the stream.  Next to a kernel launched without the attribute plain stream order holds.  The
// fp32 step (512 x 256 x 4096, nine launches then) takes 81 us with it, 99 without.
//
// Kernels of more than kPdlFlops (about a millisecond) are launched without it: there is nothing to
// gain next to their length, and placed on the SMs in the order these fall free their blocks ran
// the text8b step (four kernels of 24 to 50 ms) 0.9 % slower than in the order of a plain launch.
constexpr double kPdlFlops = 2e12;

inline cudaLaunchAttribute pdl_attribute(double flops = 0.0) {
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = flops < kPdlFlops ? 1 : 0;
  return a;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_sized(double flops, void (*kern)(KArgs...), dim3 grid, dim3 block,
                             size_t smem, cudaStream_t s, const Args&... args) {
  cudaLaunchAttribute attr[1] = {pdl_attribute(flops)};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       const Args&... args) {
  return launch_pdl_sized(0.0, kern, grid, block, smem, s, args...);
}

}  // namespace alr
