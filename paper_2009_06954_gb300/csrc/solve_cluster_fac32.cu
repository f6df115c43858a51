// Instantiations of the cluster-scope solve (solve_cluster.cuh): the incomplete factor, inner solves in FP32.
#include "solve_cluster.cuh"

namespace asss {

template asss_status cl_dispatch<float, 3, 512>(const Ctx&, const ClArgs<float>&, int, int, int, int*);

}  // namespace asss
