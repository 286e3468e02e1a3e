// Cluster forms of the FP64 march and of the pipelined step (march.cuh, Hooks::kCluster): one
// simulation, or one beam step, per cluster of 2, 4 or 8 CTAs of 256 threads, for launches with
// fewer simulations (steps) than the GPU has SMs.  One template set, instantiated per precision
// form (march_cluster_mixed.cu, march_cluster_fp64.cu).  The mixed plain marches have none: sums
// over a cluster are another order of their deposits (march.cuh, kPlain).
#pragma once

#include <mutex>

#include "march_launch.h"
#include "pipeline.cuh"

namespace wake {

constexpr int kClNT = 256;

inline int cluster_ppt(int np, int cn) {
  const int per = (np + cn - 1) / cn, ppt = (per + kClNT - 1) / kClNT;
  return ppt <= 1 ? 1 : ppt <= 2 ? 2 : ppt <= 4 ? 4 : ppt <= 8 ? 8 : 0;
}

// kMarch: the form has cluster marches, not steps only.
template <class P, bool kMarch = true>
struct ClusterForm {
  using C = ClusterOf<P>;
  using S = SlabOf<ClusterOf<P>>;

  template <int PPT>
  static size_t smem(bool step, int n1) {
    return step ? step_smem_bytes<C, kClNT, PPT>(n1) : MarchSmem<C>::bytes(n1, kClNT * PPT);
  }
  static size_t smem_of(bool step, int n1, int ppt) {
    switch (ppt) {
      case 1: return smem<1>(step, n1);
      case 2: return smem<2>(step, n1);
      case 4: return smem<4>(step, n1);
      case 8: return smem<8>(step, n1);
      default: return (size_t)1 << 40;
    }
  }
  template <class Q, int PPT>
  static const void *kernel_of(bool step) {
    if constexpr (kMarch)
      if (!step) return (const void *)march_cluster_kernel<Q, kClNT, PPT>;
    return (const void *)step_cluster_kernel<Q, kClNT, PPT>;
  }
  template <class Q>
  static const void *kernel(bool step, int ppt) {
    switch (ppt) {
      case 1: return kernel_of<Q, 1>(step);
      case 2: return kernel_of<Q, 2>(step);
      case 4: return kernel_of<Q, 4>(step);
      default: return kernel_of<Q, 8>(step);
    }
  }
  // The kernel for np rings on n1 nodes in clusters of cn, its shared-memory limit raised (the
  // limit only grows: a call that finds it high enough makes no CUDA call, so a step can be captured
  // once it was prepared).  Null when none fits.
  static const void *prepare(bool slab, bool step, int n1, int np, int cn, size_t *bytes, cudaError_t *err) {
    *err = cudaSuccess;
    const int ppt = cluster_ppt(np, cn);
    *bytes = smem_of(step, n1, ppt);
    if ((!step && !kMarch) || ppt == 0 || n1 > C::kScanE * kClNT || *bytes > kMaxSmemPerCta) return nullptr;
    const void *k = slab ? kernel<S>(step, ppt) : kernel<C>(step, ppt);
    static std::mutex mu;
    static size_t set[2][2][4] = {};
    size_t &cur = set[slab][step][ppt == 1 ? 0 : ppt == 2 ? 1 : ppt == 4 ? 2 : 3];
    std::lock_guard<std::mutex> lk(mu);
    if (*bytes > cur) {
      *err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*bytes);
      if (*err != cudaSuccess) return nullptr;
      cur = *bytes;
    }
    return k;
  }
  // Clusters of cn that the GPU holds at once (0: the form does not fit).
  static int max_clusters(bool slab, bool step, int n1, int np, int cn) {
    size_t bytes;
    cudaError_t e;
    const void *k = prepare(slab, step, n1, np, cn, &bytes, &e);
    if (!k) return 0;
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at[2];
    cluster_config(&c, at, 1, cn, kClNT, bytes, false, nullptr);
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, k, &c) == cudaSuccess ? n : 0;
  }
  static cudaError_t launch(bool slab, bool step, int n1, int np, int cn, int clusters, void **args, cudaStream_t stream) {
    size_t bytes;
    cudaError_t e;
    const void *k = prepare(slab, step, n1, np, cn, &bytes, &e);
    if (!k) return e != cudaSuccess ? e : cudaErrorInvalidValue;
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at[2];
    cluster_config(&c, at, clusters, cn, kClNT, bytes, step, stream);
    return cudaLaunchKernelExC(&c, k, args);
  }
};

}  // namespace wake
