// Launchers of the tensor-core GEMM of the backward products (plain_gemm_kernel.cuh): the
// single-CTA form, built here; the cluster forms are launched through libalr_cluster.so
// (cluster_forms.h).
#include <atomic>

#include "launch.h"
#include "plain_gemm_kernel.cuh"

namespace alr {
namespace {

// Launch configuration of a split-K cluster of n_cta CTAs (attr, two entries, must outlive the
// launch).
cudaLaunchConfig_t split_config(cudaLaunchAttribute* attr, int n_cta, int n_tiles, cudaStream_t s) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(n_cta);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(n_cta) * unsigned(n_tiles));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = s;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

template <class Kern>
cudaError_t split_attributes(Kern kern) {
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

template <typename Elem, bool kAMN, bool kBMN, bool kAcc>
cudaError_t launch_split_t(const CUtensorMap& a, const CUtensorMap& b, const GemmArgs& args,
                           cudaStream_t s) {
  auto kern = plain_gemm_kernel<Elem, kAMN, kBMN, kAcc, SplitCluster>;
  cudaError_t e = split_attributes(kern);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = split_config(attr, args.split, args.n_tiles, s);
  return cudaLaunchKernelEx(&cfg, kern, a, b, args);
}

template <typename Elem, bool kAMN, bool kBMN, bool kAcc>
cudaError_t launch_t(const CUtensorMap& a, const CUtensorMap& b, const GemmArgs& args,
                     cudaStream_t s) {
  if (args.split > 1) return launch_split_t<Elem, kAMN, kBMN, kAcc>(a, b, args, s);
  auto kern = plain_gemm_kernel<Elem, kAMN, kBMN, kAcc, NoCluster>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes));
  if (e != cudaSuccess) return e;
  return launch_pdl_sized(args.flops(), kern, args.grid, kThreads, kSmemBytes, s, a, b, args);
}

template <typename Elem>
cudaError_t dispatch(bool a_mn, bool b_mn, bool acc, const CUtensorMap& a, const CUtensorMap& b,
                     const GemmArgs& args, cudaStream_t s) {
  if constexpr (sizeof(Elem) == 4) {
    // tf32 products take K-major operands only
    if (a_mn || b_mn) return cudaErrorInvalidValue;
    return acc ? launch_t<Elem, false, false, true>(a, b, args, s)
               : launch_t<Elem, false, false, false>(a, b, args, s);
  } else {
    const int key = (a_mn ? 4 : 0) | (b_mn ? 2 : 0) | (acc ? 1 : 0);
    switch (key) {
      case 0: return launch_t<Elem, false, false, false>(a, b, args, s);
      case 1: return launch_t<Elem, false, false, true>(a, b, args, s);
      case 2: return launch_t<Elem, false, true, false>(a, b, args, s);
      case 3: return launch_t<Elem, false, true, true>(a, b, args, s);
      case 4: return launch_t<Elem, true, false, false>(a, b, args, s);
      case 5: return launch_t<Elem, true, false, true>(a, b, args, s);
      case 6: return launch_t<Elem, true, true, false>(a, b, args, s);
      default: return launch_t<Elem, true, true, true>(a, b, args, s);
    }
  }
}

}  // namespace

int plain_gemm_split_clusters(int n_cta) {
  // per-device occupancy, computed once per size (concurrent first calls compute the same value)
  static std::atomic<int> cached[64][kMaxSplit + 1];
  int dev = 0;
  if (n_cta < 2 || n_cta > kMaxSplit || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
    return 0;
  const int known = cached[dev][n_cta].load(std::memory_order_relaxed);
  if (known != 0) return known > 0 ? known : 0;
  auto kern = plain_gemm_kernel<__nv_bfloat16, false, false, false, SplitCluster>;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = split_config(attr, n_cta, 1, nullptr);
  int n = 0;
  if (split_attributes(kern) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();   // a size the device cannot place: not an error of the call
    n = 0;
  }
  cached[dev][n_cta].store(n > 0 ? n : -1, std::memory_order_relaxed);
  return n;
}

cudaError_t launch_plain_gemm(int dtype, bool a_mn, bool b_mn, bool accumulate,
                              const CUtensorMap& a, const CUtensorMap& b, const GemmArgs& args,
                              cudaStream_t s) {
  if (dtype == 0) return dispatch<__nv_bfloat16>(a_mn, b_mn, accumulate, a, b, args, s);
  return dispatch<float>(a_mn, b_mn, accumulate, a, b, args, s);
}

}  // namespace alr
