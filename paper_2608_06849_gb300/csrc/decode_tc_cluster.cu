// The cluster split of the tcgen05 decode (decode_tc.cuh, kCluster).
#include <mutex>

#include "decode_tc.cuh"

namespace aoh {

cudaError_t launch_decode_tc_cluster(const DecodeArgs& a, int cluster, cudaStream_t s) {
  return dtc::launch_mode<128, dtc::kCluster>(a, cluster, s);
}

// Clusters of `size` CTAs (one an SM) that the current device runs at once.
int decode_tc_max_clusters(int size) {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static int known[kDevices][dec::kClusterMax + 1] = {};
  int dev = 0;
  if (size < 1 || size > dec::kClusterMax || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return 0;
  std::lock_guard<std::mutex> lock(mu);
  int& n = known[dev][size];
  if (n == 0) {
    constexpr int smem = dtc::Lay<128, 1>::SMEM;
    auto kernel = dtc::decode_tc_kernel<128, 1, dtc::kCluster>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size * 64);
    cfg.blockDim = dim3(dtc::kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = -1;
    }
  }
  return n > 0 ? n : 0;
}

}  // namespace aoh
