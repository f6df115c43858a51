// Instantiations of the persistent mrs solve (mrs_kernel.cuh): skew diagonals, FP32 (Q in FP32 and BF16).
#include "mrs_kernel.cuh"

namespace asss {

template asss_status dispatch_kp<float, 1>(ASSS_MRS_DISPATCH_ARGS(float));
template asss_status dispatch_kp16<1>(ASSS_MRS_DISPATCH16_ARGS);

}  // namespace asss
