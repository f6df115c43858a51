// Instantiations of the persistent mrs solve (mrs_kernel.cuh): SELL-C storage.
#include "mrs_kernel.cuh"

namespace asss {

template asss_status dispatch_kp<float, 0>(ASSS_MRS_DISPATCH_ARGS(float));
template asss_status dispatch_kp<double, 0>(ASSS_MRS_DISPATCH_ARGS(double));
template asss_status dispatch_kp16<0>(ASSS_MRS_DISPATCH16_ARGS);

}  // namespace asss
