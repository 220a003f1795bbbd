// The H2Share reuse step's instances of the tcgen05 decode kernel (a unit of
// their own, so that the library's units compile side by side).
#include "decode_tc.cuh"

namespace aoh {

cudaError_t launch_decode_tc_reuse(const DecodeArgs& a, cudaStream_t s) { return dtc::launch_mode<128, dtc::kGather>(a, 1, s); }

}  // namespace aoh
