// Rules of the solve path that need no CUDA, so that any host can check them.
#pragma once

#include <cstdint>

#include "asss.h"

namespace asss {

// Whether the single-column solve takes the row stream (DStream) for n rows with nnz entries off the
// diagonal, vectors of tbytes a value.  The vector stays below 192 KB, which leaves the block its partial
// sums and row sums, and its indices below 16 bits.  From 64 entries a row on, half of a warp's lanes
// or more have an entry in the row's first load; below that SELL's lane per row wastes less.
// Offsets are 32-bit: a matrix whose rows, padded by up to 3 entries each, may pass them stays in SELL.
inline bool stream_fits(int n, int64_t nnz, int tbytes) {
    return (int64_t)n * tbytes <= 192000 && nnz >= (int64_t)64 * n && nnz + 3LL * n < (1LL << 31) - 1024;
}

// what a whole-solve launch reports of a column; block 0 writes it before the column's last barrier
struct ClStat {
    int outer_its, cycles, status, solves, op_calls, orth_calls;
    long long inner_its, orth_vecs;
    unsigned long long ns_inner, ns_op, ns_orth;
    double relres;
    unsigned phase;   // grid scope: barriers passed on the counter
};
constexpr int CL_CHUNK = 16;   // columns of a launch
struct ClReport {
    int wait;   // grid scope: the barrier's status word, ASSS_ERR_TIMEOUT from any block that gave up
    ClStat st[CL_CHUNK];
};

// Whether an FP32 solve on skew diagonals is faster in grid scope than launch by launch.  A large
// solve's launches cost little beside its steps, and k_mrs has more registers for them: at 130^3
// (2.2 * 10^6 rows), k = 12 / 16 / 20 / 24, grid 3366 / 3308 / 3289 / 3341 us, launches 3210 / 3399 / 3439 / 3294;
// at 150^3 (3.4 * 10^6) 4829 / 4767 / 4858 / 5055 and 4447 / 4705 / 4867 / 4753.  Without deflation, whose
// rows have the fewest loads: 100^3 1125 / 1300, 115^3 1673 / 1700, 130^3 2937 / 2548, 150^3 4128 / 3387.
inline bool grid_scope_pays(int n, int kp) { return n <= (kp > 0 ? 2500000 : 1600000); }

// rounds that nrhs columns take when `side` of them are solved side by side, in launches of CL_CHUNK
inline int cl_waves(int nrhs, int side) {
    const int rest = nrhs % CL_CHUNK;
    return nrhs / CL_CHUNK * ((CL_CHUNK + side - 1) / side) + (rest + side - 1) / side;
}

// before a launch of nc columns: nothing is reported yet, so that what the kernel does not get to
// write (the columns after a wait that ran out) does not pass for an earlier launch's result
inline void cl_expect(ClReport& r, int nc) {
    r.wait = ASSS_OK;
    for (int t = 0; t < nc; ++t) r.st[t].status = ASSS_ERR_TIMEOUT;
}

// after it: ASSS_ERR_TIMEOUT when any wait ran out, also one at a column's last barrier, where
// that column's own status says nothing; *phase: barriers passed on the counter, 0 when the
// counter has to be cleared before the next launch
inline asss_status cl_outcome(const ClReport& r, int nc, unsigned* phase) {
    *phase = 0;
    if (r.wait != ASSS_OK) return ASSS_ERR_TIMEOUT;
    for (int t = 0; t < nc; ++t)
        if (r.st[t].status == ASSS_ERR_TIMEOUT) return ASSS_ERR_TIMEOUT;
    *phase = r.st[nc - 1].phase;
    return ASSS_OK;
}

}  // namespace asss
