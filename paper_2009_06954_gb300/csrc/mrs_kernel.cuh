// Persistent single-kernel mrs solve (paper §3.1, App. B) of
//     (shift I + sign * (J~ - Q_k S_k Q_k^T)) x = b
// with J~ exactly skew - stored as skew half-diagonals (stencil-like patterns), in
// SELL-C, read in place as CSR, or applied in factored form L~^-1 J^ L~^-T through the
// incomplete L D L^T (one grid barrier per colour of each triangular solve) - and
// Q_k, S_k the skew-Lanczos data of §3.2 (Fig. 2).  One cooperative launch runs the
// whole iteration:
//
//   per iteration j (one pass over the rows owned by each block):
//     y_{j+1} = sign*(nu_j J~ y_j - Q (S_k h_j)) + beta_{j-1} nu_{j-1} y_{j-1}
//       (y_j = beta_{j-1} q_j is the unnormalised Lanczos vector, nu_j = 1/beta_{j-1},
//        h_j = Q^T q_j)
//     partial sums of ||y_{j+1}||^2 and Q^T y_{j+1}   -> ONE grid-wide reduction
//     the p/x update of step j-1 (needs only scalars known before the pass)
//   then every block computes the same Givens scalars from the reduced sums:
//     theta_j = sqrt(theta~_j^2 + beta_j^2), c_j, s_j, delta_j = -s_{j-1} beta_j,
//     theta~_{j+1} = c_{j-1} theta_j, x-coefficient g_j c_j, g_{j+1} = -g_j s_j.
//
// The norm and the k deflation dot products share the single reduction per
// iteration, which keeps the method's one-synchronisation-per-step property (§3.1).
// Vectors produced by other blocks are read through L2 (ld.global.cg); the grid
// barrier has a bounded wait.
#pragma once

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include <cuda_bf16.h>

#include "common.cuh"
#include "internal.h"
#include "mrs_dev.cuh"

namespace asss {


constexpr int MRS_TRACE_STEPS = 16;
constexpr int MRS_TRACE_SLOTS = 4 + 5 * MRS_TRACE_STEPS;
// One block per SM.  512 threads: up to 128 registers a thread, which keep the loads of a
// whole row (all diagonals unrolled) in flight; more resident warps with half the
// registers measured slower (the FP32 pass is bound by memory latency per row).  The FP64
// solve on diagonals or CSR is bound by the FP64 pipe instead (2 FMAs a clock and SM, so a
// warp instruction holds it for 16 cycles): 8 warps keep it busy, and every warp that
// takes part costs its share of FP64 adds in the block's partial sums.
template <class T, int FMT>
constexpr int mrs_threads() { return sizeof(T) == 8 && (FMT == 1 || FMT == 2 || FMT == 5) ? 256 : MRS_THREADS; }

// Blocks of a launch.  FP32 (and the SELL / factored FP64 passes): one slice per warp before
// another block is opened.  The FP64-pipe-bound passes instead open a block per slice up
// to one per SM, so that the rows of a small system (n = 822..5000 in the paper) use every
// SM's FP64 pipe: a slice costs about 70 + 31 warp instructions of 16 cycles on its SM,
// one more block only one more 16-cycle add in every block's cross-block sum.  Measured with
// the folded sums (warp_fold): a step at n = 64^3, k = 20 takes 41 us instead of 68 (its
// 71 FMAs a row need 32), at n = 2209 9 us instead of 34.
template <class T, int FMT>
inline int mrs_blocks(int sms, int occ, int nslices) {
    if (mrs_threads<T, FMT>() != MRS_THREADS) occ = 1;
    const int need = mrs_threads<T, FMT>() != MRS_THREADS ? nslices : cdiv(nslices, MRS_WARPS);
    const int most = sms * (occ > 4 ? 4 : occ);
    return need < 1 ? 1 : need < most ? need : most;
}

struct MrsWork {
    int n = 0;
    const int* skip = nullptr;  // device flag read by the next launches (see mrs_set_skip)
    int sms = 0;
    DBuf<double> Y64, P64;
    DBuf<float> Y32, P32;
    DBuf<double> part;
    DBuf<unsigned> bar;
    DBuf<int> err;
    DBuf<int> out_its;
    DBuf<double> out_ratio;
    DBuf<int> blk_slice;
    const void* part_key = nullptr;
    int part_nblk = 0;
    int halo32 = -1, halo64 = -1;  // halo of the current Y layout (-1: not laid out)
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // deferred statistics: each launch writes its step count and ratio into a log
    // slot and is bracketed by its own event pair; mrs_collect reads them all at once
    static constexpr int LOG_CAP = 1024;
    DBuf<int> its_log;
    DBuf<double> ratio_log;
    std::vector<cudaEvent_t> evs;
    std::vector<long long> log_nnz, log_per_row;  // bytes model per launch
    int log_n = 0;
    MrsTotals tot;
    DBuf<unsigned long long> trace;  // ASSS_TRACE_MRS=1: timeline of block 0
    ~MrsWork() {
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        for (cudaEvent_t e : evs) cudaEventDestroy(e);
    }
};

template <class T>
struct MrsParams {
    int n;
    // SELL-C operator (rowmap: slot -> row for SELL-C-sigma, null for the identity)
    const int* sptr;
    const int* col;
    const T* val;
    const int* rowmap;
    const int4* units;   // SELL work units (slice, part, parts, accumulator) and their offsets per slice
    const int* uoff;
    T* hacc;             // partial sums of the parts of long slices (32 per long slice, left at 0)
    unsigned* hcnt;      // parts finished per long slice (left at 0)
    int split;           // entries per lane of one work unit
    // row-stream operator
    const int* rrp;
    const unsigned short* rcol;
    const T* rval;
    int racc;            // row sums held in shared memory (the most rows a block owns)
    // skew half-diagonal operator: U points at U_0[0]; diagonal d starts ustride later
    int ndiag;
    const int* off;
    const T* U;
    long long ustride;
    // plain CSR operator read in place (64-bit row pointers), one thread per row
    const long long* crp;
    const int* cci;
    const T* cval;
    // factored operator: z = wd .* (I + L)^-1 J^ (I + L)^-T (wd .* y), colour by colour
    int ncol;
    const int* fls;      // ncol + 1 level offsets into flvl
    const int* flvl;     // vertices by (colour, index)
    const int *flrp, *flci, *furp, *fuci, *fjrp, *fjci;
    const T *flv, *fuv, *fjv, *fwd;
    const int* fpart;    // 2x2 pivots: partner of each vertex (null: 1x1 pivots only)
    const T* fwo;        // off-diagonal of |D|^-1/2 between the members of a pair
    T* ft;               // (I + L)^-T (wd .* y)
    T* fw;               // (I + L)^-1 J^ ft
    long long ystride;  // distance between the three Y slots (n + 2 halo)
    long long pstride;  // distance between the two P slots
    const T* Q;
    const __nv_bfloat16* Q16;  // BF16 copy of Q (row stride KP) when the kernel reads Q in BF16
    const double* alpha;
    int k;
    double shift, sign;
    const double* rhs;
    T* x;
    T* Y;  // 3 slots of unnormalised Lanczos vectors, each with a zero halo on both ends
    T* P;  // ring of two update directions
    double* part;  // [2][NV][nblk]
    GridBarrier gb;
    const int* blk_slice;
    double tol;
    int maxit;
    long long budget;
    int* out_its;
    double* out_ratio;
    unsigned long long* trace;  // optional timeline (block 0): %globaltimer at phase boundaries
    const int* skip;     // optional: when *skip != 0 at launch the kernel only logs its = -1
    int qcs;             // load Q rows evict-first (the step's data exceed L2)
    double* qtz;         // optional: Q^T x (k values) of the final iterate
};

// sum over q in [q0, q1) of v[q] * x[ci[q]], eight entries at a time: the indices
// and values of a batch are loaded first, then all its gathers, so a row costs a
// few memory latencies instead of two per entry (x is written by other blocks of
// the launch: plain loads after the grid barrier, not the read-only path)
template <class T>
__device__ __forceinline__ T row_dot8(const int* __restrict__ ci, const T* __restrict__ v, const T* x, int q0,
                                      int q1) {
    T a = (T)0;
    for (int q = q0; q < q1; q += 8) {
        int cc[8];
        T vv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool in = q + u < q1;
            cc[u] = in ? __ldg(ci + q + u) : 0;
            vv[u] = in ? __ldg(v + q + u) : (T)0;
        }
        T g[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = (q + u < q1) ? x[cc[u]] : (T)0;
#pragma unroll
        for (int u = 0; u < 8; ++u) a += vv[u] * g[u];
    }
    return a;
}

// the products of one warp of the row-stream pass: entries [e, e1), which start in row r
// (rp: the block's row offsets, in shared memory).  Sums of rows that start here go to
// acc[row], the sum of a row that began in an earlier warp to carry / crow.
template <class T>
__device__ __forceinline__ void stream_rows(const T* __restrict__ val, const unsigned short* __restrict__ col,
                                            const T* __restrict__ y, const int* rp, int r, int e, int e1, bool cs,
                                            T* acc, T& carry, int& crow) {
    constexpr int U = sizeof(T) == 4 ? 4 : 2;   // groups of 4 entries in flight per lane and batch
    constexpr int V = sizeof(T) / 4;            // 16-byte loads of the 4 values
    struct Batch {
        int4 v[U][V];
        uint2 c[U];
    };
    const int lane = threadIdx.x & 31;
    if (e >= e1) return;
    const int first = e;
    auto load = [&](int from, int end, Batch& B) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = from + u * 128 + lane * 4;
            if (q < end) {
                const int4* vp = reinterpret_cast<const int4*>(val + q);
                const uint2* cp = reinterpret_cast<const uint2*>(col + q);
#pragma unroll
                for (int t = 0; t < V; ++t) B.v[u][t] = cs ? __ldcs(vp + t) : __ldg(vp + t);
                B.c[u] = cs ? __ldcs(cp) : __ldg(cp);
            }
        }
    };
    int end = min(rp[r + 1], e1);
    Batch cur, nxt;
    load(e, end, cur);
    T sum = (T)0;
    while (true) {
        // the batch after this one, possibly in a later row
        int ne = e + U * 128, nr = r, nend = end;
        const bool rowdone = ne >= end;
        if (rowdone) {
            ne = end;
            nr = r + 1;
            if (ne < e1) {
                while (rp[nr + 1] == ne) ++nr;   // rows without entries
                nend = min(rp[nr + 1], e1);
            }
        }
        if (ne < e1) load(ne, nend, nxt);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (e + u * 128 + lane * 4 < end) {
                const unsigned c01 = cur.c[u].x, c23 = cur.c[u].y;
                const T* v = reinterpret_cast<const T*>(cur.v[u]);
                sum += v[0] * y[c01 & 0xffffu];
                sum += v[1] * y[c01 >> 16];
                sum += v[2] * y[c23 & 0xffffu];
                sum += v[3] * y[c23 >> 16];
            }
        }
        if (rowdone) {
            const T t = warp_sum(sum);
            if (lane == 0) {
                if (rp[r] >= first) {
                    acc[r] = t;
                } else {
                    carry = t;
                    crow = r;
                }
            }
            sum = (T)0;
            if (ne >= e1) break;
        }
        cur = nxt;
        e = ne;
        r = nr;
        end = nend;
    }
}

// FMT 0: SELL-C storage of J~; FMT 1: skew half-diagonal storage; FMT 2: plain CSR;
// FMT 3: factored J~ = L~^-1 J^ L~^-T (incomplete L D L^T in a multicolour order)
// FMT 5: as FMT 1, four lanes a row (FP64 systems of at most a slice per SM).  A warp's FP64
// operation holds its SM quarter's pipe for 64 cycles whatever its lanes do, so a row a lane
// costs a warp 71 + 23 of them in a chain on one quarter of one SM; four lanes a row put a
// slice on all four quarters, at 29 + 6 each (a step at n = 2209, k = 20: 9.1 -> 6.2 us with the
// sums below).
// FMT 4: row-stream storage.  Long rows (hundreds of entries, some thousands): with a lane
// per row (SELL) a system of 2 10^4 rows has fewer work units than the GPU has warps and each
// is one lane's serial chain of gathers.  Here a block's entries are cut evenly over its 16
// warps, a warp reads a row 128 entries at a time (512 + 256 contiguous bytes) with the next
// batch already in flight, and gathers from a copy of y in shared memory; the sums of the
// rows that a cut splits are added in warp order.  Bound: L2 bandwidth of the stream (6 bytes
// an entry in FP32) and the bank conflicts of the gathers.
template <class T, int KP, int FMT, bool QB = false>
__global__ void __launch_bounds__((mrs_threads<T, FMT>()), 1) k_mrs(MrsParams<T> p) {
    constexpr int NV = KP + 1;
    constexpr bool QBLK = q_blocked<T>(FMT == 1 || FMT == 3);
    constexpr int NT = mrs_threads<T, FMT>(), NW = NT / 32;
    // x is read with a row's first loads; not in the FP64 SELL pass, where 16 entries in flight and
    // 2 (k + 1) values fill the registers and one more row value cuts the batch (n = 30 000, k = 20:
    // 286 us a step against 236; at k = 8 190 against 198)
    constexpr bool XEARLY = !(FMT == 0 && sizeof(T) == 8 && KP > 12);
    if (p.skip && *p.skip) {  // enqueued ahead of a decision that went the other way
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *p.out_its = -1;
            *p.out_ratio = 0.0;
        }
        return;
    }
    __shared__ T s_wsum[NW][NV];
    // cross-block sums: rows of partials summed by a warp each (FP32) or by groups of NV threads
    constexpr int NG = sizeof(T) == 4 ? NW : (NT / NV > 0 ? NT / NV : 1);
    __shared__ typename std::conditional<sizeof(T) == 4, float2, double>::type s_bsum[NG][NV];
    __shared__ T s_red[NV];
    __shared__ T s_u[KP > 0 ? KP : 1];
    constexpr bool DIA = FMT == 1 || FMT == 5;
    __shared__ int s_off[DIA ? MRS_MAXDIAG : 1];
    __shared__ int s_ls[FMT == 3 ? ILDL_MAXCOL + 1 : 1];
    __shared__ MrsScalars<T> sc;
    __shared__ T s_alpha[MRS_KPMAX];
    // per-step coefficients in T, set by one thread (the others only read them):
    // 0 sign*nu, 1 sign, 2 beta_{j-1} nu_{j-1}, 3 nu_p, 4 delta_pp, 5 1/theta_p, 6 xcoef_p,
    // 7..10 the final pass: nu, delta, 1/theta, xcoef
    __shared__ T s_cf[12];
    __shared__ int s_next;   // SELL: next work unit of this block for the warp that asks (see next_slice)
    // Q^T x of the final iterate without a pass over Q: the directions obey
    // p_j = (nu_j y_j - delta_j p_{j-2}) / theta_j and x = sum_j xcoef_j p_j, so Q^T p_j and
    // Q^T x follow from the Q^T y_j that every step reduces anyway (warp 1 keeps them)
    __shared__ T s_qty[KP > 0 ? KP : 1];     // Q^T y_j of the step in progress
    __shared__ T s_qtp[2][KP > 0 ? KP : 1];  // Q^T p of the last two directions (slot j & 1)
    __shared__ T s_qtx[KP > 0 ? KP : 1];     // Q^T x
    __shared__ T s_pq[4];                    // step j: nu_j, delta, 1/theta_j, xcoef_j
    if constexpr (DIA) {
        for (int d = threadIdx.x; d < p.ndiag; d += NT) s_off[d] = p.off[d];
    }
    for (int m = threadIdx.x; m < KP; m += NT) {
        s_qtp[0][m] = (T)0;
        s_qtp[1][m] = (T)0;
        s_qtx[m] = (T)0;
    }
    if constexpr (FMT == 3) {
        for (int c = threadIdx.x; c <= p.ncol; c += NT) s_ls[c] = p.fls[c];
        __syncthreads();
    }
    for (int m = threadIdx.x; m + 1 < p.k && m < MRS_KPMAX; m += NT) s_alpha[m] = (T)p.alpha[m];
    auto set_coefs = [&]() {  // thread 0 only
        s_cf[0] = (T)p.sign * sc.nu;
        s_cf[1] = (T)p.sign;
        s_cf[2] = (T)sc.coef_old;
        s_cf[3] = (T)sc.nu_p;
        s_cf[4] = (T)sc.delta_pp;
        s_cf[5] = (T)sc.rtheta_p;
        s_cf[6] = (T)sc.xcoef_p;
        if (sc.stop) {
            s_cf[7] = (T)sc.fin_nu;
            s_cf[8] = (T)sc.fin_delta;
            s_cf[9] = (T)sc.fin_rtheta;
            s_cf[10] = (T)sc.fin_xcoef;
        }
    };
    const int nblk = gridDim.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // FMT 4: the block's rows [rb, re); its slices are cut from there
    const int rb = FMT == 4 ? p.blk_slice[blockIdx.x] : 0, re = FMT == 4 ? p.blk_slice[blockIdx.x + 1] : 0;
    const int s0 = FMT == 4 ? 0 : p.blk_slice[blockIdx.x];
    const int s1 = FMT == 4 ? (re - rb + 31) >> 5 : p.blk_slice[blockIdx.x + 1];
    const int n = FMT == 4 ? re : p.n;   // the end of this block's rows
    const size_t ys = p.ystride;
    // timeline slots: 0 start, 1 phase-0 pass, 2 phase-0 barrier, 3 set-up scalars; then per
    // step j (1-based, first MRS_TRACE_STEPS): 4+5(j-1)+{0 pass, 1 partials, 2 barrier, 3 reduce, 4 scalars+u}
    const bool tr = p.trace && blockIdx.x == 0 && threadIdx.x == 0;
    auto stamp = [&](int slot) {
        if (tr && slot < MRS_TRACE_SLOTS) p.trace[slot] = gtimer();
    };
    stamp(0);

    // warp sums in T, then across the warps that hold rows in a fixed order (float pairs for
    // the FP32 solve, FP64 for the FP64 solve) into this block's partials
    using P2 = typename std::conditional<sizeof(T) == 4, float2, double>::type;
    auto add = [](P2 a, P2 b) {
        if constexpr (sizeof(T) == 4) return df_add(a, b);
        else return a + b;
    };
    const int nact0 = FMT == 0 ? NW : min(NW, max(s1 - s0, 1));
    const int nact5 = min(NW, max(4 * (s1 - s0), 1));   // FMT 5: a warp takes a quarter of a slice
    auto block_partials = [&](T(&tacc)[NV], double* buf, bool quarters) {
        const int nact = quarters ? nact5 : nact0;
        if (warp < nact) {
            if (FMT == 5 && quarters) {
                // lane (row r, part q): tacc[0] the norm's share, tacc[1 + t] the sum of
                // column q + 4 t; summed over the eight rows, three exchanges
                constexpr int TV = KP / 4 + 1;
                T v[TV];
#pragma unroll
                for (int t = 0; t < TV; ++t) v[t] = tacc[t];
                int idx = 0, have = TV, cnt = TV;
#pragma unroll
                for (int o = 16; o >= 4; o >>= 1) {
                    const bool up = (lane & o) != 0;
                    const int h = (cnt + 1) / 2;
#pragma unroll
                    for (int i = 0; i < (TV + 1) / 2; ++i)
                        if (i < h) {
                            const T lo = v[i], hi = h + i < cnt ? v[h + i < TV ? h + i : 0] : (T)0;
                            v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
                        }
                    idx += up ? h : 0;
                    have = up ? have - h : min(have, h);
                    cnt = h;
                }
                // up to TV / 8 rounded up values are left a lane (one for k <= 28)
#pragma unroll
                for (int i = 0; i < (TV + 7) / 8; ++i)
                    if (i < have) {
                        const int t = idx + i, q = lane & 3;
                        if (t > 0) s_wsum[warp][1 + q + 4 * (t - 1)] = v[i];
                        else if (q == 0) s_wsum[warp][0] = v[i];
                    }
            } else {
                warp_fold_to<NV>(tacc, s_wsum[warp]);
            }
        }
        __syncthreads();
        for (int v = threadIdx.x; v < NV; v += NT) {
            if constexpr (sizeof(T) == 4) {
                // block partial as a float pair (hi, lo) in the same 8 bytes
                float2 a[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) a[w] = make_float2(w < nact ? s_wsum[w][v] : 0.f, 0.f);
                reinterpret_cast<float2*>(buf)[(size_t)blockIdx.x * NV + v] = pair_tree(a, add);
            } else {
                double a[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) a[w] = w < nact ? s_wsum[w][v] : 0.0;
                buf[(size_t)blockIdx.x * NV + v] = pair_tree(a, add);
            }
        }
    };
    // every block adds the block partials in the same fixed order: warp w takes blocks
    // w, w + NW, ..., a lane one value (a block's values are contiguous; the loads of
    // RCHUNK blocks are in flight together), then warp 0 adds the warps' sums into s_red.
    // Only warp 0 holds s_red afterwards: it goes on with the scalars (FP64: every warp).
    constexpr int RCHUNK = 10;
    auto reduce_all = [&](const double* buf) {
        if constexpr (sizeof(T) == 8) {
            // FP64: the adds are what this costs (64 cycles a warp and SM quarter), so every
            // lane takes one: thread g NV + v the value v of blocks g, g + NG, ...; then four
            // lanes a value
            for (int t = threadIdx.x; t < NG * NV; t += NT) {
                const int v = t % NV, g = t / NV;
                double acc = 0.0;
                for (int b0 = g; b0 < nblk; b0 += NG * RCHUNK) {
                    double ld[RCHUNK];
#pragma unroll
                    for (int q = 0; q < RCHUNK; ++q) {
                        const int b = b0 + q * NG;
                        ld[q] = b < nblk ? __ldcg(&buf[(size_t)b * NV + v]) : 0.0;
                    }
#pragma unroll
                    for (int q = 0; q < RCHUNK; ++q)
                        if (b0 + q * NG < nblk) acc += ld[q];
                }
                s_bsum[g][v] = acc;
            }
            __syncthreads();
            for (int t0 = 0; t0 < 4 * NV; t0 += NT) {
                const int t = t0 + threadIdx.x, v = t >> 2;
                double a = 0.0;
                if (v < NV)
                    for (int g = t & 3; g < NG && g < nblk; g += 4) a += s_bsum[g][v];
                a += __shfl_xor_sync(0xffffffffu, a, 1);
                a += __shfl_xor_sync(0xffffffffu, a, 2);
                if (v < NV && (t & 3) == 0) s_red[v] = a;
            }
            __syncthreads();
            return;
        }
        const P2* b2 = reinterpret_cast<const P2*>(buf);
        for (int v = lane; v < NV; v += 32) {
            P2 acc{};
            for (int b0 = warp; b0 < nblk; b0 += NW * RCHUNK) {
                P2 ld[RCHUNK];
#pragma unroll
                for (int t = 0; t < RCHUNK; ++t) {
                    const int b = b0 + t * NW;
                    ld[t] = b < nblk ? __ldcg(&b2[(size_t)b * NV + v]) : P2{};
                }
#pragma unroll
                for (int t = 0; t < RCHUNK; ++t)
                    if (b0 + t * NW < nblk) acc = add(acc, ld[t]);   // (warp-uniform)
            }
            s_bsum[warp][v] = acc;
        }
        __syncthreads();
        if (warp == 0) {
            for (int v = lane; v < NV; v += 32) {
                P2 ws[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) ws[w] = s_bsum[w][v];
                const P2 a = pair_tree(ws, add);
                if constexpr (sizeof(T) == 4) s_red[v] = a.x + a.y;
                else s_red[v] = a;
            }
            __syncwarp();
        }
    };
    // square roots and their reciprocals of two numbers at once, a in lane 0 and b in lane 1
    // (two dependent chains side by side; FP64 through rsqrt, whose chain is the shortest)
    auto roots = [&](T a, T b, T& ra, T& ia, T& rb, T& ib) {
        const T rad = lane == 0 ? a : b;
        T root, inv;
        if constexpr (sizeof(T) == 4) {
            root = sqrt(rad);
            inv = (T)1 / root;
        } else {
            inv = rsqrt(rad);
            root = rad != (T)0 ? rad * inv : (T)0;
        }
        ra = __shfl_sync(0xffffffffu, root, 0);
        ia = __shfl_sync(0xffffffffu, inv, 0);
        rb = __shfl_sync(0xffffffffu, root, 1);
        ib = __shfl_sync(0xffffffffu, inv, 1);
    };
    // u = S_k h with h = nu * (Q^T y), S_k(m, m+1) = alpha_m, S_k(m+1, m) = -alpha_m;
    // computed by the lanes of warp 0 (the caller synchronises the block afterwards)
    auto make_u_warp0 = [&](T nu) {
        if constexpr (KP > 0) {
            for (int m = lane; m < KP; m += 32) {
                T u = (T)0;
                if (m < p.k) {
                    if (m + 1 < p.k) u += s_alpha[m] * s_red[2 + m] * nu;
                    if (m > 0) u -= s_alpha[m - 1] * s_red[m] * nu;
                }
                s_u[m] = u;
            }
        }
    };
    // warp 1: fold direction p_jj into Q^T x (s_pq holds step jj's scalars, s_qty Q^T y_jj)
    auto qtx_fold = [&](int jj) {
        if constexpr (KP > 0) {
#pragma unroll
            for (int m = lane; m < lane + KP; m += 32) {   // two values a lane above k = 32
                if (m < p.k) {
                    T* pp = s_qtp[jj & 1];
                    const T v = (s_pq[0] * s_qty[m] - s_pq[1] * pp[m]) * s_pq[2];
                    pp[m] = v;
                    s_qtx[m] += s_pq[3] * v;
                }
            }
        }
    };
    const bool want_qtx = KP > 0 && p.qtz != nullptr;
    unsigned phase = 0;  // grid barriers passed in this launch
    // row-stream storage: this warp's entries [e0, e1) of the block's, from row wr on, and in
    // dynamic shared memory y, the block's row sums and row offsets
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ T s_carry[FMT == 4 ? NW : 1];
    __shared__ int s_crow[FMT == 4 ? NW : 1];
    T* s_y = reinterpret_cast<T*>(s_dyn);
    T* s_acc = s_y + ((p.n + 3) & ~3);
    int* s_rp = reinterpret_cast<int*>(s_acc + p.racc);
    int e0 = 0, e1 = 0, wr = 0;
    if constexpr (FMT == 4) {
        const int nr = re - rb;
        for (int t = threadIdx.x; t <= nr; t += NT) s_rp[t] = __ldg(&p.rrp[rb + t]);
        __syncthreads();
        const int chunk = ((s_rp[nr] - s_rp[0] + NW - 1) / NW + 127) & ~127;
        e0 = min(s_rp[0] + warp * chunk, s_rp[nr]);
        e1 = min(e0 + chunk, s_rp[nr]);
        int lo = 0, hi = nr;   // the last row that starts at or before e0
        while (lo < hi) {
            const int mid = lo + ((hi - lo + 1) >> 1);
            if (s_rp[mid] <= e0) lo = mid;
            else hi = mid - 1;
        }
        wr = lo;
    }
    // ---- phase 0: y_1 = b, x = 0, p = 0, ||b||^2 and Q^T b ----
    T tacc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) tacc[v] = (T)0;
    // The slices of a SELL operator carry very different amounts of work (heavy-tailed
    // rows), so in the step passes the warps of a block take them one at a time from a
    // shared counter instead of in a fixed stride; the other storages keep the stride.
    auto next_slice = [&](int sl) -> int {
        if constexpr (FMT == 0) {
            int nx = 0;
            if (lane == 0) nx = atomicAdd(&s_next, 1);
            return __shfl_sync(0xffffffffu, nx, 0);
        }
        return sl + NW;
    };
    // SELL: the block's work units (its slices, long ones cut into parts)
    const int u0 = FMT == 0 ? __ldg(&p.uoff[s0]) : s0;
    const int u1 = FMT == 0 ? __ldg(&p.uoff[s1]) : s1;
    // the row held by lane `lane` of slice sl (SELL-C-sigma permutes rows within windows)
    auto row_of = [&](int sl) -> int {
        if constexpr (FMT == 0) {
            if (p.rowmap) return __ldg(&p.rowmap[sl * 32 + lane]);
        }
        return rb + sl * 32 + lane;
    };
    for (int sl = s0 + warp; sl < s1; sl += NW) {
        int i = row_of(sl);
        if (i < n) {
            T b = (T)p.rhs[i];
            p.Y[i] = b;
            p.x[i] = (T)0;
            p.P[i] = (T)0;
            p.P[p.pstride + i] = (T)0;
            tacc[0] += b * b;
            T q[KP > 0 ? KP : 1];
            if constexpr (QB) load_qrow16<T, KP>(p.Q16, i, q);
            else load_qrow<T, KP, QBLK>(p.Q, i, q, p.qcs != 0);
#pragma unroll
            for (int m = 0; m < KP; ++m) tacc[1 + m] += q[m] * b;
        }
    }
    stamp(1);
    block_partials(tacc, p.part, false);
    const bool met = grid_sync_phase(p.gb, nblk, phase++, p.budget);
    stamp(2);
    if (!met) return;
    reduce_all(p.part);

    if (warp == 0) {
        if (lane == 0) {
            const T r0 = sqrt(s_red[0]);
            const T zero = (T)0, one = (T)1;
            sc.r0 = r0;
            sc.rr0 = r0 > zero ? one / r0 : zero;
            sc.nu = sc.rr0;
            sc.coef_old = zero;
            sc.theta_t = (T)p.shift;
            sc.c_prev = one;
            sc.s_prev = zero;
            sc.delta_prev = zero;
            sc.G = r0;
            sc.nu_p = zero;
            sc.delta_pp = zero;
            sc.rtheta_p = one;
            sc.xcoef_p = zero;
            sc.ratio = r0 > zero ? one : zero;
            sc.its = 0;
            sc.stop = r0 > zero ? 0 : 1;
            set_coefs();
            s_next = u0 + NW;
        }
        __syncwarp();
        if (!sc.stop) make_u_warp0(sc.nu);
    }
    __syncthreads();
    if (sc.stop) {  // b = 0: x = 0 already
        if (blockIdx.x == 0) {
            if (threadIdx.x == 0) {
                *p.out_its = 0;
                *p.out_ratio = 0.0;
            }
            if (p.qtz)
                for (int v = threadIdx.x; v < p.k; v += NT) p.qtz[v] = 0.0;
        }
        return;
    }
    stamp(3);

    for (int j = 1; j <= p.maxit; ++j) {
        const int tb = 4 + 5 * (j - 1);
        if (want_qtx && warp == 1) {
            // off the synchronisation chain: step j-1's direction, then Q^T y_j from the
            // last reduction (s_red is next written after this pass's block barrier)
            if (j >= 2) qtx_fold(j - 1);
#pragma unroll
            for (int m = lane; m < lane + KP; m += 32)
                if (m < p.k) s_qty[m] = s_red[1 + m];
        }
        // the step's vectors do not overlap: restrict lets later rows' loads be scheduled
        // ahead of this row's stores
        const T* __restrict__ Ycur = p.Y + (size_t)((j - 1) % 3) * ys;
        const T* __restrict__ Yold = p.Y + (size_t)((j + 1) % 3) * ys;
        T* __restrict__ Ynew = p.Y + (size_t)(j % 3) * ys;
        T* __restrict__ Pj1 = p.P + (size_t)((j - 1) & 1) * p.pstride;
        T* __restrict__ xv = p.x;
        const T* __restrict__ Ub = p.U;
        const T* __restrict__ Qr = p.Q;
        const T tnu = s_cf[0], tsg = s_cf[1], tco = s_cf[2];
        const T tnp = s_cf[3], tdpp = s_cf[4], tthp = s_cf[5], txp = s_cf[6];
        if constexpr (FMT == 3) {
            // J~ y_j in factored form: the back solve (I + L)^T t = wd .* y_j from the
            // largest colour down, then w = (I + L)^-1 J^ t from the smallest colour up
            // (J^ t is formed row by row inside the forward solve); the rows of one
            // colour are spread over the whole grid, one grid barrier per colour
            const int gt = blockIdx.x * NT + threadIdx.x, gs = nblk * NT;
            bool ok = true;
            for (int cc = p.ncol - 1; cc >= 0 && ok; --cc) {
                for (int e = s_ls[cc] + gt; e < s_ls[cc + 1]; e += gs) {
                    const int i = __ldg(&p.flvl[e]);
                    T a = __ldg(&p.fwd[i]) * Ycur[i];
                    if (p.fpart) {
                        const int m = __ldg(&p.fpart[i]);
                        if (m >= 0) a += __ldg(&p.fwo[i]) * Ycur[m];
                    }
                    p.ft[i] = a - row_dot8<T>(p.fuci, p.fuv, p.ft, __ldg(&p.furp[i]), __ldg(&p.furp[i + 1]));
                }
                ok = grid_sync_phase(p.gb, nblk, phase++, p.budget);
            }
            for (int cc = 0; cc < p.ncol && ok; ++cc) {
                for (int e = s_ls[cc] + gt; e < s_ls[cc + 1]; e += gs) {
                    const int i = __ldg(&p.flvl[e]);
                    const T a = row_dot8<T>(p.fjci, p.fjv, p.ft, __ldg(&p.fjrp[i]), __ldg(&p.fjrp[i + 1]));
                    p.fw[i] = a - row_dot8<T>(p.flci, p.flv, p.fw, __ldg(&p.flrp[i]), __ldg(&p.flrp[i + 1]));
                }
                ok = grid_sync_phase(p.gb, nblk, phase++, p.budget);
            }
            if (!ok) break;
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) tacc[v] = (T)0;
        // a row once its product with J~ is there: y_{j+1}, its sums, the p/x update of step j-1
        auto finish = [&](int i, T acc, T yold, T pold, T xold, T(&q)[KP > 0 ? KP : 1]) {
            T dq = (T)0;
#pragma unroll
            for (int m = 0; m < KP; ++m) dq += q[m] * s_u[m];
            T ynew = tnu * acc - tsg * dq + tco * yold;
            Ynew[i] = ynew;
            tacc[0] += ynew * ynew;
#pragma unroll
            for (int m = 0; m < KP; ++m) tacc[1 + m] += q[m] * ynew;
            if (j >= 2) {
                T pv = (tnp * yold - tdpp * pold) * tthp;
                Pj1[i] = pv;
                xv[i] = (XEARLY ? xold : xv[i]) + txp * pv;
            }
        };
        if constexpr (FMT == 4) {
            auto qrow = [&](int i, T(&q)[KP > 0 ? KP : 1]) {
                if constexpr (QB) load_qrow16<T, KP>(p.Q16, i, q);
                else load_qrow<T, KP, QBLK>(Qr, i, q, p.qcs != 0);
            };
            // the first row's own data, in flight during the products
            int i = rb + threadIdx.x;
            T q[KP > 0 ? KP : 1], yold = (T)0, pold = (T)0, xold = (T)0;
            if (i < re) {
                if (j >= 2) {
                    yold = Yold[i];
                    pold = Pj1[i];
                    xold = xv[i];
                }
                qrow(i, q);
            }
            // y into shared memory (every slot starts on 16 bytes and is padded to 16)
            constexpr int VW = 16 / sizeof(T);
            const int4* yv4 = reinterpret_cast<const int4*>(Ycur);
            int4* sy4 = reinterpret_cast<int4*>(s_y);
            const int nv4 = (p.n + VW - 1) / VW;
#pragma unroll 8
            for (int t = threadIdx.x; t < nv4; t += NT) sy4[t] = yv4[t];
            for (int t = threadIdx.x; t < re - rb; t += NT) s_acc[t] = (T)0;
            if (threadIdx.x < NW) s_crow[threadIdx.x] = -1;
            __syncthreads();
            stream_rows<T>(p.rval, p.rcol, s_y, s_rp, wr, e0, e1, p.qcs != 0, s_acc, s_carry[warp], s_crow[warp]);
            __syncthreads();
            for (; i < re; i += NT) {
                T acc = s_acc[i - rb];
#pragma unroll
                for (int w = 0; w < NW; ++w)
                    if (s_crow[w] == i - rb) acc += s_carry[w];
                finish(i, acc, yold, pold, xold, q);
                if (i + NT < re) {
                    if (j >= 2) {
                        yold = Yold[i + NT];
                        pold = Pj1[i + NT];
                        xold = xv[i + NT];
                    }
                    qrow(i + NT, q);
                }
            }
        } else if constexpr (FMT == 5) {
            const int sub = lane & 3;
            for (int qq = 4 * s0 + warp; qq < 4 * s1; qq += NW) {
                const int i = qq * 8 + (lane >> 2);
                const bool live = i < n;
                T part = (T)0, q[KP > 0 ? KP / 4 : 1], yold = (T)0, pold = (T)0;
                if (live) {
                    if (j >= 2) {
                        yold = Yold[i];
                        if (sub == 0) pold = Pj1[i];
                    }
                    const T* qr = Qr + (size_t)i * KP + sub;
#pragma unroll
                    for (int t = 0; t < KP / 4; ++t) q[t] = __ldg(qr + 4 * t);
                    const T* Ud = Ub + i;
                    const T* yi = Ycur + i;
                    T acc = (T)0, dq = (T)0;
#pragma unroll 3
                    for (int d = sub; d < p.ndiag; d += 4) {
                        const int m = s_off[d];
                        const T* Um = Ud + d * p.ustride;
                        acc = fma(__ldg(Um), yi[m], acc);
                        acc = fma(-__ldg(Um - m), yi[-m], acc);
                    }
#pragma unroll
                    for (int t = 0; t < KP / 4; ++t) dq += q[t] * s_u[sub + 4 * t];
                    part = tnu * acc - tsg * dq;
                }
                part += __shfl_xor_sync(0xffffffffu, part, 1);
                part += __shfl_xor_sync(0xffffffffu, part, 2);
                if (live) {
                    const T ynew = part + tco * yold;
#pragma unroll
                    for (int t = 0; t < KP / 4; ++t) tacc[1 + t] += q[t] * ynew;
                    if (sub == 0) {
                        Ynew[i] = ynew;
                        tacc[0] += ynew * ynew;
                        if (j >= 2) {
                            const T pv = (tnp * yold - tdpp * pold) * tthp;
                            Pj1[i] = pv;
                            xv[i] += txp * pv;
                        }
                    }
                }
            }
        } else {
        for (int uu = u0 + warp; uu < u1; uu = next_slice(uu)) {
            int sl = uu, part = 0, nparts = 1, hix = -1;
            if constexpr (FMT == 0) {
                const int4 U = __ldg(&p.units[uu]);
                sl = U.x;
                part = U.y;
                nparts = U.z;
                hix = U.w;
            }
            const int i = row_of(sl);
            const bool live = i < n;
            // this row's own data first (independent of the operator loop below)
            const T yold = (live && j >= 2) ? Yold[i] : (T)0;
            const T pold = (live && j >= 2) ? Pj1[i] : (T)0;
            // x with the other loads ahead of the products: read at its use, its latency stood
            // at the end of every row (FP32 pass at 100^3: 26.4 -> 24.5 us, at 47^3 3.55 -> 3.33)
            const T xold = (XEARLY && live && j >= 2) ? xv[i] : (T)0;
            uint4 qraw[(QB && KP > 0) ? KP / 8 : 1];
            if constexpr (QB && KP > 0) {
                if (live) {
                    const uint4* qr = reinterpret_cast<const uint4*>(p.Q16 + (size_t)i * KP);
#pragma unroll
                    for (int t = 0; t < KP / 8; ++t) qraw[t] = p.qcs ? __ldcs(qr + t) : __ldg(qr + t);
                }
            }
            T acc = (T)0;
            if constexpr (FMT == 3) {
                if (live) {
                    acc = __ldg(&p.fwd[i]) * p.fw[i];
                    if (p.fpart) {
                        const int m = __ldg(&p.fpart[i]);
                        if (m >= 0) acc += __ldg(&p.fwo[i]) * p.fw[m];
                    }
                }
            } else if constexpr (FMT == 2) {
                if (i < n) {
                    const long long e1 = __ldg(&p.crp[i + 1]);
                    for (long long e = __ldg(&p.crp[i]); e < e1; ++e) acc += __ldg(&p.cval[e]) * Ycur[__ldg(&p.cci[e])];
                }
            } else if constexpr (FMT == 0) {
                const int base = __ldg(&p.sptr[sl]);
                const int wfull = (__ldg(&p.sptr[sl + 1]) - base) >> 5;
                // this unit's part of the slice: entries [part * split, ...) of every lane
                const int kbeg = part * p.split;
                const int width = min(wfull, kbeg + p.split) - kbeg;
                const int* cp = p.col + base + lane + kbeg * 32;
                const T* vp = p.val + base + lane + kbeg * 32;
                // Sixteen entries in flight per lane (the gathers depend on the column
                // loads, so the depth of the batch is the latency hiding); when the
                // matrix exceeds L2 its entries are loaded evict-first, so the gathered
                // vector stays in L2 while the matrix streams past it.
                constexpr int UB = 16;
                int kk = 0;
                if (p.qcs) {
                    for (; kk + UB <= width; kk += UB) {
                        int cc[UB];
                        T vv[UB];
#pragma unroll
                        for (int u = 0; u < UB; ++u) {
                            cc[u] = __ldcs(cp + (kk + u) * 32);
                            vv[u] = __ldcs(vp + (kk + u) * 32);
                        }
#pragma unroll
                        for (int u = 0; u < UB; ++u) acc += vv[u] * Ycur[cc[u]];
                    }
                    for (; kk < width; ++kk) acc += __ldcs(vp + kk * 32) * Ycur[__ldcs(cp + kk * 32)];
                } else {
                    for (; kk + UB <= width; kk += UB) {
                        int cc[UB];
                        T vv[UB];
#pragma unroll
                        for (int u = 0; u < UB; ++u) {
                            cc[u] = __ldg(cp + (kk + u) * 32);
                            vv[u] = __ldg(vp + (kk + u) * 32);
                        }
#pragma unroll
                        for (int u = 0; u < UB; ++u) acc += vv[u] * Ycur[cc[u]];
                    }
                    for (; kk < width; ++kk) acc += __ldg(vp + kk * 32) * Ycur[__ldg(cp + kk * 32)];
                }
                if (nparts > 1) {
                    // a part of a long slice: add the lanes' partial sums; the warp that
                    // finishes the slice's last part reads the totals (resetting them for
                    // the next pass) and carries on with the rows, the others are done
                    atomicAdd(&p.hacc[(size_t)hix * 32 + lane], acc);
                    __threadfence();
                    __syncwarp();
                    int last = 0;
                    if (lane == 0) last = atomicAdd(&p.hcnt[hix], 1u) == (unsigned)(nparts - 1);
                    last = __shfl_sync(0xffffffffu, last, 0);
                    if (!last) continue;
                    __threadfence();
                    // every other part's adds completed before its count (fenced), and no
                    // one touches this slice's accumulators again before the next pass
                    acc = __ldcg(&p.hacc[(size_t)hix * 32 + lane]);
                    p.hacc[(size_t)hix * 32 + lane] = (T)0;
                    if (lane == 0) p.hcnt[hix] = 0u;
                }
            } else {
                // (J~ y)_i = sum_d U_d[i] y[i + m_d] - U_d[i - m_d] y[i - m_d]; zero halos on
                // both U (front) and y (both ends) make the loop branch-free
                if (i < n) {
                    const T* Ud = Ub + i;
                    const T* yi = Ycur + i;
                    if constexpr (sizeof(T) == 4) {
                        acc = dia_row<T, 12>(Ud, p.ustride, yi, s_off, p.ndiag);
                    } else {
#pragma unroll 12
                        for (int d = 0; d < p.ndiag; ++d, Ud += p.ustride) {
                            const int m = s_off[d];   // two FMAs a diagonal, no separate product and sum
                            acc = fma(__ldg(Ud), yi[m], acc);
                            acc = fma(-__ldg(Ud - m), yi[-m], acc);
                        }
                    }
                }
            }
            if (live) {
                T q[KP > 0 ? KP : 1];
                if constexpr (QB && KP > 0) {
#pragma unroll
                    for (int t = 0; t < KP / 8; ++t) {
                        const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&qraw[t]);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float2 f = __bfloat1622float2(h2[e]);
                            q[8 * t + 2 * e] = (T)f.x;
                            q[8 * t + 2 * e + 1] = (T)f.y;
                        }
                    }
                } else {
                    load_qrow<T, KP, QBLK>(Qr, i, q, p.qcs != 0);
                }
                finish(i, acc, yold, pold, xold, q);
            }
        }
        }
        double* buf = p.part + (size_t)(j & 1) * NV * nblk;
        stamp(tb);
        block_partials(tacc, buf, FMT == 5);
        stamp(tb + 1);
        const bool met = grid_sync_phase(p.gb, nblk, phase++, p.budget);
        stamp(tb + 2);
        if (!met) break;
        reduce_all(buf);
        stamp(tb + 3);

        if (warp == 0) {
            T beta, rbeta, theta, rth;
            roots(s_red[0], sc.theta_t * sc.theta_t + s_red[0], beta, rbeta, theta, rth);
            if (lane == 0) {
                const T c = sc.theta_t * rth, s = beta * rth;
                const T delta = -sc.s_prev * beta;
                const T theta_t_next = sc.c_prev * theta;
                const T xcoef = sc.G * c;
                const T Gn = -sc.G * s;
                s_pq[0] = sc.nu;
                s_pq[1] = sc.delta_prev;
                s_pq[2] = rth;
                s_pq[3] = xcoef;
                sc.ratio = fabs(Gn) * sc.rr0;
                sc.its = j;
                if (sc.ratio < p.tol || j == p.maxit) {
                    sc.stop = 1;
                    sc.fin_nu = sc.nu;
                    sc.fin_delta = sc.delta_prev;
                    sc.fin_rtheta = rth;
                    sc.fin_xcoef = xcoef;
                } else {
                    sc.nu_p = sc.nu;
                    sc.delta_pp = sc.delta_prev;
                    sc.rtheta_p = rth;
                    sc.xcoef_p = xcoef;
                    sc.coef_old = beta * sc.nu;
                    sc.nu = (beta != (T)0) ? rbeta : (T)0;
                    sc.s_prev = s;
                    sc.c_prev = c;
                    sc.delta_prev = delta;
                    sc.theta_t = theta_t_next;
                    sc.G = Gn;
                }
                set_coefs();
                s_next = u0 + NW;
            }
            if constexpr (sizeof(T) == 4) {
                __syncwarp();
                if (!sc.stop) make_u_warp0(sc.nu);
            }
        } else if (sizeof(T) == 8 && warp == 2) {
            // FP64: u on another quarter of the SM, beside the scalars (unused after a stop)
            make_u_warp0(s_red[0] != (T)0 ? (T)rsqrt((double)s_red[0]) : (T)0);
        }
        __syncthreads();
        if (sc.stop) {
            T* Pj = p.P + (size_t)(j & 1) * p.pstride;
            const T tn = s_cf[7], td = s_cf[8], tth = s_cf[9], tx = s_cf[10];
#pragma unroll
            for (int v = 0; v < NV; ++v) tacc[v] = (T)0;
            for (int sl = s0 + warp; sl < s1; sl += NW) {
                int i = row_of(sl);
                if (i < n) {
                    T pv = (tn * Ycur[i] - td * Pj[i]) * tth;
                    p.x[i] = p.x[i] + tx * pv;
                }
            }
            if (want_qtx && warp == 1) {
                qtx_fold(j);
                if (blockIdx.x == 0) {
#pragma unroll
                    for (int m = lane; m < lane + KP; m += 32)
                        if (m < p.k) p.qtz[m] = (double)s_qtx[m];
                }
            }
            break;
        }
        stamp(tb + 4);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *p.out_its = sc.its;
        *p.out_ratio = (double)sc.ratio;
    }
}

// what the launcher needs to know about the operator, whatever its storage
template <class T>
struct OpView {
    int n = 0;
    int fmt = 0;
    int nslices = 0;
    const int* sptr = nullptr;
    const int* col = nullptr;
    const T* val = nullptr;
    const int* rowmap = nullptr;
    const int4* units = nullptr;
    const int* uoff = nullptr;
    T* hacc = nullptr;
    unsigned* hcnt = nullptr;
    int nheavy = 0;
    int split = 0;
    int ndiag = 0;
    const int* off = nullptr;
    const T* U = nullptr;
    long long ustride = 0;
    int halo = 0;
    const void* key = nullptr;
    long long nnz = 0;  // matrix entries one application reads
    const IldlFactor* fac = nullptr;  // FMT 3
    const int* rrp = nullptr;         // FMT 4
    const unsigned short* rcol = nullptr;
    const T* rval = nullptr;
    long long rstored = 0;
};

struct LaunchOut {
    int slot;
    double* qtz;
};

template <class T, int KP, int FMT, bool QB = false>
static asss_status launch_mrs(const Ctx& c, MrsWork* w, const OpView<T>& J, const T* Q, const double* alpha,
                              int k, double shift, double sign, const double* rhs, T* x, T* Y, long long ystride,
                              T* P, double tol, int maxit, LaunchOut lo, const __nv_bfloat16* Q16 = nullptr) {
    // row-stream storage: a row weighs its entries plus what its own data cost, so that a
    // block owns at most (total weight / blocks) / that cost + 2 rows, whose sums and offsets
    // stand in shared memory behind y
    int rowcost = 0, racc = 0, smem = 0;
    if constexpr (FMT == 4) {
        rowcost = (int)std::max<long long>(48, J.rstored / J.n / 8);
        racc = (int)((J.rstored + (long long)rowcost * J.n) / ((long long)rowcost * std::min(c.sms, J.n))) + 4;
        racc = (racc + 3) & ~3;
        smem = (int)(sizeof(T) * (((long long)J.n + 3) / 4 * 4 + racc) + sizeof(int) * (racc + 1));
        ASSS_TRY(raise_dynamic_smem((const void*)k_mrs<T, KP, FMT, QB>, smem));
    }
    int occ = 0;
    ASSS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mrs<T, KP, FMT, QB>, (mrs_threads<T, FMT>()),
                                                            smem));
    if (occ < 1) {
        set_error("mrs kernel cannot be resident");
        return ASSS_ERR_CUDA;
    }
    // (FMT 5: a slice a block, by the rule that chose it)
    const int nblk = FMT == 4 ? std::min(c.sms, J.n) : mrs_blocks<T, FMT>(c.sms, occ, J.nslices);
    if (w->part_key != J.key || w->part_nblk != nblk) {
        if (FMT == 4)
            k_partition_rows<<<cdiv(nblk + 1, 128), 128, 0, c.stream>>>(J.rrp, J.n, rowcost, nblk, w->blk_slice.p);
        else
            k_partition<<<cdiv(nblk + 1, 128), 128, 0, c.stream>>>(FMT == 0 ? J.sptr : nullptr, J.nslices, nblk,
                                                                   w->blk_slice.p);
        ASSS_CHECK_LAUNCH();
        w->part_key = J.key;
        w->part_nblk = nblk;
    }
    ASSS_CUDA(cudaMemsetAsync(w->bar.p, 0, 2 * sizeof(unsigned), c.stream));
    if (FMT == 0 && J.nheavy > 0) {
        // the long slices' accumulators start at zero (a launch that gave up at a barrier
        // may have left partial sums behind)
        ASSS_CUDA(cudaMemsetAsync(J.hacc, 0, sizeof(T) * 32 * (size_t)J.nheavy, c.stream));
        ASSS_CUDA(cudaMemsetAsync(J.hcnt, 0, sizeof(unsigned) * (size_t)J.nheavy, c.stream));
    }
    MrsParams<T> prm;
    prm.n = J.n;
    prm.sptr = J.sptr;
    prm.col = J.col;
    prm.val = J.val;
    prm.rowmap = J.rowmap;
    prm.units = J.units;
    prm.uoff = J.uoff;
    prm.hacc = J.hacc;
    prm.hcnt = J.hcnt;
    prm.split = J.split > 0 ? J.split : SELL_SPLIT;
    prm.ndiag = J.ndiag;
    prm.off = J.off;
    prm.U = J.U;
    prm.ustride = J.ustride;
    prm.rrp = J.rrp;
    prm.rcol = J.rcol;
    prm.rval = J.rval;
    prm.racc = racc;
    prm.crp = nullptr;
    prm.cci = nullptr;
    prm.cval = nullptr;
    prm.ncol = 0;
    prm.fls = prm.flvl = prm.flrp = prm.flci = prm.furp = prm.fuci = prm.fjrp = prm.fjci = nullptr;
    prm.flv = prm.fuv = prm.fjv = prm.fwd = nullptr;
    prm.fpart = nullptr;
    prm.fwo = nullptr;
    prm.ft = prm.fw = nullptr;
    if constexpr (FMT == 3) {
        const IldlFactor& F = *J.fac;
        prm.ncol = F.ncol;
        prm.fpart = F.npairs > 0 ? F.part.p : nullptr;
        prm.fls = F.ls.p;
        prm.flvl = F.lvl.p;
        prm.flrp = F.lrp.p;
        prm.flci = F.lci.p;
        prm.furp = F.urp.p;
        prm.fuci = F.uci.p;
        prm.fjrp = F.jrp;
        prm.fjci = F.jci;
        if constexpr (sizeof(T) == 4) {
            prm.flv = F.lv32.p;
            prm.fuv = F.uv32.p;
            prm.fjv = F.jv32.p;
            prm.fwd = F.wd32.p;
            prm.fwo = F.wo32.p;
            prm.ft = F.ft32.p;
            prm.fw = F.fw32.p;
        } else {
            prm.flv = F.lv.p;
            prm.fuv = F.uv.p;
            prm.fjv = F.jv;
            prm.fwd = F.wd.p;
            prm.fwo = F.wo.p;
            prm.ft = F.ft.p;
            prm.fw = F.fw.p;
        }
    }
    prm.ystride = ystride;
    prm.pstride = pad32(J.n);
    prm.Q = Q;
    prm.Q16 = Q16;
    prm.alpha = alpha;
    prm.k = k;
    prm.shift = shift;
    prm.sign = sign;
    prm.rhs = rhs;
    prm.x = x;
    prm.Y = Y;
    prm.P = P;
    prm.part = w->part.p;
    prm.gb.count = w->bar.p;
    prm.gb.err = w->err.p;
    prm.blk_slice = w->blk_slice.p;
    prm.tol = tol;
    prm.maxit = maxit;
    prm.budget = c.wait_cycles;
    prm.out_its = w->its_log.p + lo.slot;
    prm.out_ratio = w->ratio_log.p + lo.slot;
    prm.qtz = (KP > 0 && k > 0) ? lo.qtz : nullptr;
    prm.trace = w->trace.p;
    prm.skip = w->skip;
    {
        const long long qrow = QB ? 2LL * KP : (long long)sizeof(T) * KP;
        prm.qcs = stream_evict_first(c, J.nnz * (long long)sizeof(T) + (long long)J.n * (7LL * sizeof(T) + qrow)) ? 1 : 0;
    }
    void* args[] = {&prm};
    ASSS_CUDA(cudaEventRecord(w->evs[2 * lo.slot], c.stream));
    ASSS_CUDA(cudaLaunchCooperativeKernel((const void*)k_mrs<T, KP, FMT, QB>, dim3(nblk), dim3(mrs_threads<T, FMT>()),
                                          args, smem, c.stream));
    count_launch();
    ASSS_CUDA(cudaEventRecord(w->evs[2 * lo.slot + 1], c.stream));
    return ASSS_OK;
}

template <class T, int FMT>
asss_status dispatch_kp(const Ctx& c, MrsWork* w, const OpView<T>& J, const T* Q, const double* alpha, int k,
                               int kp, double shift, double sign, const double* rhs, T* x, T* Y, long long ystride,
                               T* P, double tol, int maxit, LaunchOut lo) {
    switch (kp) {
#define ASSS_MRS_CASE(KPV) \
    case KPV:              \
        return launch_mrs<T, KPV, FMT>(c, w, J, Q, alpha, k, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
        ASSS_MRS_CASE(0)
        ASSS_MRS_CASE(4)
        ASSS_MRS_CASE(8)
        ASSS_MRS_CASE(12)
        ASSS_MRS_CASE(16)
        ASSS_MRS_CASE(20)
        ASSS_MRS_CASE(24)
        ASSS_MRS_CASE(32)
        ASSS_MRS_CASE(48)
        ASSS_MRS_CASE(64)
#undef ASSS_MRS_CASE
        default:
            set_error("unsupported padded Lanczos width %d", kp);
            return ASSS_ERR_UNSUPPORTED;
    }
}

// FP32 solve reading Q in BF16: row strides that keep 16-byte aligned rows
template <int FMT>
asss_status dispatch_kp16(const Ctx& c, MrsWork* w, const OpView<float>& J, const __nv_bfloat16* Q16,
                                 const double* alpha, int k, int kp, double shift, double sign, const double* rhs,
                                 float* x, float* Y, long long ystride, float* P, double tol, int maxit,
                                 LaunchOut lo) {
    switch (kp) {
#define ASSS_MRS16_CASE(KPV) \
    case KPV:                \
        return launch_mrs<float, KPV, FMT, true>(c, w, J, nullptr, alpha, k, shift, sign, rhs, x, Y, ystride, P, tol, \
                                                 maxit, lo, Q16);
        ASSS_MRS16_CASE(8)
        ASSS_MRS16_CASE(16)
        ASSS_MRS16_CASE(24)
        ASSS_MRS16_CASE(32)
        ASSS_MRS16_CASE(48)
        ASSS_MRS16_CASE(64)
#undef ASSS_MRS16_CASE
        default:
            set_error("unsupported BF16 Lanczos width %d", kp);
            return ASSS_ERR_UNSUPPORTED;
    }
}

#define ASSS_MRS_DISPATCH_ARGS(T)                                                                                    \
    const Ctx&, MrsWork*, const OpView<T>&, const T*, const double*, int, int, double, double, const double*, T*,    \
        T*, long long, T*, double, int, LaunchOut
#define ASSS_MRS_DISPATCH16_ARGS                                                                                     \
    const Ctx&, MrsWork*, const OpView<float>&, const __nv_bfloat16*, const double*, int, int, double, double,       \
        const double*, float*, float*, long long, float*, double, int, LaunchOut
// instantiated in mrs_dia32.cu, mrs_dia64.cu, mrs_sell.cu, mrs_stream.cu and mrs_fac.cu, which
// build in parallel
extern template asss_status dispatch_kp<float, 0>(ASSS_MRS_DISPATCH_ARGS(float));
extern template asss_status dispatch_kp<float, 1>(ASSS_MRS_DISPATCH_ARGS(float));
extern template asss_status dispatch_kp<float, 3>(ASSS_MRS_DISPATCH_ARGS(float));
extern template asss_status dispatch_kp<double, 0>(ASSS_MRS_DISPATCH_ARGS(double));
extern template asss_status dispatch_kp<double, 1>(ASSS_MRS_DISPATCH_ARGS(double));
extern template asss_status dispatch_kp<double, 5>(ASSS_MRS_DISPATCH_ARGS(double));
extern template asss_status dispatch_kp<double, 3>(ASSS_MRS_DISPATCH_ARGS(double));
extern template asss_status dispatch_kp<float, 4>(ASSS_MRS_DISPATCH_ARGS(float));
extern template asss_status dispatch_kp<double, 4>(ASSS_MRS_DISPATCH_ARGS(double));
extern template asss_status dispatch_kp16<4>(ASSS_MRS_DISPATCH16_ARGS);
extern template asss_status dispatch_kp16<0>(ASSS_MRS_DISPATCH16_ARGS);
extern template asss_status dispatch_kp16<1>(ASSS_MRS_DISPATCH16_ARGS);

}  // namespace asss
