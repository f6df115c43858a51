// Instantiations of the persistent mrs solve (mrs_kernel.cuh): row-stream storage.
#include "mrs_kernel.cuh"

namespace asss {

template asss_status dispatch_kp<float, 4>(ASSS_MRS_DISPATCH_ARGS(float));
template asss_status dispatch_kp<double, 4>(ASSS_MRS_DISPATCH_ARGS(double));
template asss_status dispatch_kp16<4>(ASSS_MRS_DISPATCH16_ARGS);

}  // namespace asss
