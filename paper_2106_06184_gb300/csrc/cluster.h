// Thread-block clusters along x: the launch configuration, and whether a device schedules one.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace sldm {

struct ClusterLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  ClusterLaunch(int cs, unsigned ctas, unsigned threads, size_t smem, cudaStream_t s) {
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(cs);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

// One kernel's answer by device.  It is asked for at the most dynamic shared memory that any launch may take: the
// small launches that come first fit where several CTAs of a cluster share an SM, and say nothing of the large ones.
struct ClusterFit {
  std::atomic<uint64_t> yes{0}, no{0};
};
inline bool cluster_fits(ClusterFit& f, int dev, const void* kernel, int cs, unsigned threads, size_t most_smem) {
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (f.yes.load() & bit) return true;
  if (f.no.load() & bit) return false;
  bool ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most_smem)) == cudaSuccess;
  if (ok && cs > 8) ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  if (ok) {
    const ClusterLaunch c(cs, unsigned(cs), threads, most_smem, 0);
    int n = 0;
    ok = cudaOccupancyMaxActiveClusters(&n, kernel, &c.cfg) == cudaSuccess && n > 0;
  }
  if (!ok) cudaGetLastError();
  (ok ? f.yes : f.no).fetch_or(bit);
  return ok;
}

}  // namespace sldm
