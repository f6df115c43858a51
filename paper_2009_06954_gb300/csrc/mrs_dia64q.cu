// Instantiations of the persistent mrs solve (mrs_kernel.cuh): skew diagonals, FP64, four
// lanes a row.
#include "mrs_kernel.cuh"

namespace asss {

template asss_status dispatch_kp<double, 5>(ASSS_MRS_DISPATCH_ARGS(double));

}  // namespace asss
