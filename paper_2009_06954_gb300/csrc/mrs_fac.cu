// Instantiations of the persistent mrs solve (mrs_kernel.cuh): the factored operator.
#include "mrs_kernel.cuh"

namespace asss {

template asss_status dispatch_kp<float, 3>(ASSS_MRS_DISPATCH_ARGS(float));
template asss_status dispatch_kp<double, 3>(ASSS_MRS_DISPATCH_ARGS(double));

}  // namespace asss
