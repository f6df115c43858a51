// Instantiations of the cluster-scope solve (solve_cluster.cuh): skew diagonals, inner solves in FP64,
// many rows a block (grid scope).
#include "solve_cluster.cuh"

namespace asss {

template asss_status cl_dispatch<double, 1, 512>(const Ctx&, const ClArgs<double>&, int, int, int, int*);

}  // namespace asss
