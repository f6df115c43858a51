// Instantiations of the cluster-scope solve (solve_cluster.cuh): skew diagonals, inner solves in FP32,
// few rows a CTA.
#include "solve_cluster.cuh"

namespace asss {

template asss_status cl_dispatch<float, 1, 256>(const Ctx&, const ClArgs<float>&, int, int, int, int*);

}  // namespace asss
