// What a context knows of the library's kernels on its device: the shared-memory attribute, set
// once, and how many clusters of each size can be resident.
#pragma once
#include <algorithm>
#include <cuda_runtime.h>
#include <vector>

namespace still {

constexpr int kMaxCluster = 8;

// A kernel that needs more dynamic shared memory than the default, or whose launch depends on how
// many clusters of cluster_lo .. cluster_hi CTAs can be resident (cluster_hi 1: no clusters).
struct KernelEntry {
  const void* fn = nullptr;
  int threads = 0, smem = 0;
  int cluster_lo = 1, cluster_hi = 1;
};

// Every such kernel of the library, in no particular order. It is filled while the library is
// loaded (KernelId) and only read afterwards.
inline std::vector<KernelEntry>& kernel_entries() {
  static std::vector<KernelEntry> entries;
  return entries;
}
inline int add_kernel(const KernelEntry& e) {
  kernel_entries().push_back(e);
  return (int)kernel_entries().size() - 1;
}

// The place of one kernel in kernel_entries(): a launcher that names KernelId<...>::value puts its
// kernel there, so that no list of instantiations has to be kept by hand.
template <auto Kernel, int kThreads, int kSmem, int kClusterLo = 1, int kClusterHi = kClusterLo>
struct KernelId {
  static_assert(kClusterHi <= kMaxCluster, "cluster size");
  static inline const int value = add_kernel(
      {reinterpret_cast<const void*>(Kernel), kThreads, kSmem, kClusterLo, kClusterHi});
};

struct KernelState {
  cudaError_t status = cudaErrorInvalidDeviceFunction;  // of setting the attribute
  int clusters[kMaxCluster + 1] = {0};                  // resident clusters by size; 0: not known
};

// The CUDA calls that fill a table (replaced by a stand-in in the tests, which need no GPU).
struct KernelQuery {
  cudaError_t (*set_smem)(const void* fn, int bytes) = [](const void* fn, int bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  cudaError_t (*clusters)(int* n, const KernelEntry& e, int size, int grid) =
      [](int* n, const KernelEntry& e, int size, int grid) {
        cudaLaunchConfig_t q = {};
        q.gridDim = dim3(grid, 1, 1);
        q.blockDim = dim3(e.threads, 1, 1);
        q.dynamicSmemBytes = e.smem;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = size;
        a[0].val.clusterDim.y = 1;
        a[0].val.clusterDim.z = 1;
        q.attrs = a;
        q.numAttrs = 1;
        return cudaOccupancyMaxActiveClusters(n, e.fn, &q);
      };
};

// One per context, filled when the context is created with its device current, and read-only
// afterwards: calls ask the driver for nothing (they may be under capture), host threads share
// nothing, and two contexts on two devices each have their own device's answers.
struct KernelTable {
  int num_sms = 0;
  std::vector<KernelState> kernels;

  void fill(int sms, const KernelQuery& query = KernelQuery()) {
    num_sms = sms;
    kernels.assign(kernel_entries().size(), KernelState());
    for (size_t i = 0; i < kernels.size(); ++i) {
      const KernelEntry& e = kernel_entries()[i];
      KernelState& k = kernels[i];
      k.status = query.set_smem(e.fn, e.smem);
      for (int c = std::max(2, e.cluster_lo); k.status == cudaSuccess && c <= e.cluster_hi; ++c) {
        int n = 0;
        if (query.clusters(&n, e, c, c * std::max(1, sms / c)) == cudaSuccess)
          k.clusters[c] = std::max(0, std::min(n, sms / c));
      }
    }
    cudaGetLastError();  // a refused query is in the table, not an error of the next launch
  }

  template <class Id>
  const KernelState& of() const {
    return kernels[Id::value];
  }
  // The grid of a persistent kernel on clusters of `size`: as many as can be resident, or one
  // per `size` SMs where that is not known.
  template <class Id>
  int persistent_clusters(int size) const {
    const int n = of<Id>().clusters[size];
    return n > 0 ? n : std::max(1, num_sms / size);
  }
};

}  // namespace still
