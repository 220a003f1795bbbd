// The d_head 64 instances of the tcgen05 decode kernel (decode_tc.cuh, Lay).
#include "decode_tc.cuh"

namespace aoh {

cudaError_t launch_decode_tc64(const DecodeArgs& a, cudaStream_t s) {
  if (a.cluster > 0) return dtc::launch_mode<64, dtc::kCluster>(a, a.cluster, s);
  return dtc::launch_mode<64, dtc::kStream>(a, 1, s);
}

}  // namespace aoh
