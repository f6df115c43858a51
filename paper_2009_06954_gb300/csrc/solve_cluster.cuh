// Whole solves in one launch, a thread-block cluster per right-hand side: the refinement loop
// on the true FP64 residual, flexible GMRES (FP64) and P^-1 by Eq. smw around the mrs
// iteration of App. B in T, the algorithms of refine / fgmres_cycle / apply_prec (asss.cu) and of
// k_mrs in cluster scope.
//
// What bounds a solve of a small or middling system in the launch-by-launch path is not its
// data but its 30 to 100 launches, the host's decisions between them and the grid-wide
// barriers inside them.  Here the CTAs of a cluster own contiguous rows; sums over the system
// are exchanged through distributed shared memory, every CTA adds them in the same order and
// takes the same decisions, and vectors that other CTAs read go through L2 around a cluster
// barrier.  Several right-hand sides are as many clusters side by side (see CL_SIZES).
// Bound: the latency of a row's loads and of a synchronisation; for larger systems a cluster's share
// of the bandwidth and of the FP64 pipe, so those run the same code in grid scope (cluster_size
// in asss.cu has both sides measured).
#pragma once

#include <algorithm>

#include "cluster_dev.cuh"
#include "internal.h"
#include "mrs_dev.cuh"
#include "solve_rules.h"

namespace asss {

constexpr int CL_RESTART = 60;           // longest restart (the Hessenberg matrix stands in shared memory)
constexpr int CL_XV = CL_RESTART + 6;    // values of one exchange
constexpr int CL_MMAX = 320;             // largest SMW rank k + r
// CTAs of a cluster to choose from.  A cluster lives in one GPC, of which this GPU has seven
// with 16 SMs to spare, eight with 12: 7, 8, 13 and 15 clusters of these sizes are resident.
constexpr int CL_NSIZES = 4;
constexpr int CL_SIZES[CL_NSIZES] = {16, 12, 10, 8};
constexpr int CL_REGV = 6;               // vectors whose dot products run together in registers

// y_i = sum_j M_ij x_j: a diagonal copy (at most 16 diagonals) or CSR
struct ClMat {
    int ndiag;
    const int* off;
    const double* val;
    const int *rp, *ci;
    const double* v;
};

// one triangle or J^ in (colour, index) order
template <class T>
struct ClRows {
    const int *rp, *ci;
    const T* v;         // in the precision of the inner solve
    const double* d;    // FP64
};
// the incomplete factor (FMT 3): colours, their rows, L, U and J^ by position, the weights
// |D|^-1/2 (wo: off-diagonals of the 2x2 pivots, part null without any)
template <class T>
struct ClFactor {
    int ncol, own_max;   // own_max: the most rows of all colours that a CTA owns (cl_run)
    const int *ls, *lvl, *pos;
    ClRows<T> L, U, J;
    const double *wd, *wo;
    const T *wdT, *woT;
    const int* part;
};

template <class T>
struct ClArgs {
    int n, ncol, restart;
    // J~ by skew diagonals (as k_mrs FMT 1), Q_k (q_blocked), S_k, SMW data
    int ndiag, halo, k, m, r;
    const int* off;
    const T* U;
    long long ustride;
    const T* Q;
    const double* alpha;
    const T* Ys;              // n x m row-major
    const int *neg, *neg2;    // U_r (UrCols of asss.cu)
    const double *negc1, *negc2;
    // op1 then op2: the outer operator; Sm and Am: update and residual (their transposes with tr)
    ClMat op1, op2, Sm, Am;
    ClFactor<T> fac;          // FMT 3
    const double *dr, *dc, *w;
    const int* perm;
    int tr;
    double sign;
    const double* b;          // column c at b + c * ldb
    long long ldb;
    double* x;
    long long ldx;
    double* work;             // per resident cluster
    long long work_stride;
    double outer_tol, inner_tol;
    int outer_maxit, inner_maxit;
    ClStat* stats;            // pinned host memory (ClReport), read after the stream is synchronised
    unsigned phase0;          // grid scope: barriers passed before this launch
    // grid scope: block partials (2 x [blocks][CL_XV]), barrier and its budget, evict-first loads of
    // what is read once (the data of a step exceed L2); the barrier's status word stands in the
    // pinned report too, so the host has it without a copy (a wait reads it every 64th poll only)
    double* part;
    GridBarrier gb;
    long long budget;
    int cs;
};

// doubles of workspace per cluster
inline long long cl_work_doubles(int n, int halo, int restart, int tbytes) {
    const long long nd = (5 + 2 * restart + 1) * pad32(n);
    const long long nt = 3 * (pad32(n) + 2LL * halo + 32) + 3 * pad32(n);
    return nd + (nt * tbytes + 7) / 8 + 64;
}

template <class T, int KP, bool GRID, int NT>
struct ClShared {
    static constexpr int NW = NT / 32;
    using P2 = typename std::conditional<sizeof(T) == 4, float2, double>::type;
    unsigned long long x[2][GRID ? 1 : CL_MAX][CL_XV];   // exchanged block sums, written by the other CTAs
    double bsum[GRID ? NT / (KP + 1) + 1 : 1][KP + 1];   // grid scope: parts of the cross-block sums
    T wsum[NW][KP + 1];
    double wd[NW][CL_REGV + 2];
    double bp[CL_XV], tot[CL_XV];
    T red[KP + 1], u[KP > 0 ? KP : 1], alpha[KP > 0 ? KP : 1], cf[12];
    T qty[KP > 0 ? KP : 1], qtp[2][KP > 0 ? KP : 1], qtx[KP > 0 ? KP : 1], pq[4];
    T wv[CL_MMAX];
    int off[64], moff[4][16];
    double h1[CL_RESTART + 1], cs[CL_RESTART + 1], sn[CL_RESTART + 1], g[CL_RESTART + 2], yv[CL_RESTART + 1];
    double fin[3];
    MrsScalars<T> sc;
    int stop;
};

// shared memory behind the Hessenberg matrix with FMT 3: the replicated vectors of the sweeps
// (two in T, or one in FP64 in the same place), and per own row its value, vertex and the
// row of L, U and J^; then the colours' first own row and first position
template <class T>
inline long long cl_factor_smem(int n, int own_max, int ncol) {
    return std::max<long long>(2LL * n * (long long)sizeof(T), 8LL * n) + 8 + (long long)own_max * (8 + 4 + 3 * 8) +
           4LL * (2 * ncol + 2);
}

constexpr size_t CL_SMEM_MAX = 227 * 1024;
// shared memory behind the `used` bytes for the rows of Q_k of a block; 0: they do not fit
inline size_t cl_q_bytes(int n, int kp, int blocks, size_t used) {
    const size_t need = 16 + 32 * 4 * (size_t)kp * cdiv(cdiv(n, 32), blocks);
    return used + need <= CL_SMEM_MAX ? need : 0;
}

// row i of Q_k, from a CTA's slices in shared memory (its first row rb) or from global memory
template <class T, int KP, bool QS>
__device__ __forceinline__ void cl_qrow(const T* __restrict__ Q, const float4* s_q, int rb, int i,
                                        T (&q)[KP > 0 ? KP : 1], bool cs) {
    if constexpr (QS) {
        const float4* a = s_q + (size_t)((i - rb) >> 5) * 8 * KP + (i & 31);
#pragma unroll
        for (int m = 0; m < KP; m += 4, a += 32) {
            const float4 v = *a;
            q[m] = v.x;
            q[m + 1] = v.y;
            q[m + 2] = v.z;
            q[m + 3] = v.w;
        }
    } else {
        load_qrow<T, KP, q_blocked<T>(true)>(Q, i, q, cs);
    }
}

// One triangular solve, colour by colour (back: from the last colour down): vec[e] =
// own[row of e] - sum_q v_q vec[col_q], vec replicated in every CTA; own: this CTA's right-hand
// side, in the order of its rows.  Four lanes share a row (an FP64 operation of a warp takes 64
// cycles, however many of its lanes work) and its stores to the other CTAs; the entries
// of the next two colours are on their way while a colour is solved.  Not inlined: its
// registers would add to the solve's, at five places.
template <class E, int NT>
__device__ __noinline__ void cl_tri_sweep(E* vec, const E* own, const int2* rows, const int* __restrict__ ci,
                                          const E* __restrict__ v, bool back, int ncol, const int* s_off,
                                          const int* s_beg) {
    constexpr int PF = 4;   // entries a lane fetches ahead
    struct Slot {
        int2 rw;
        int cc[PF];
        E vv[PF];
    };
    const int tid = threadIdx.x, sub = tid & 3;
    const unsigned C = cl_size();
    auto fetch = [&](int o, int end, Slot& S) {
        S.rw = o < end ? rows[o] : make_int2(0, 0);
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int q = sub + 4 * u;
            S.cc[u] = q < S.rw.y ? __ldg(ci + S.rw.x + q) : 0;
            S.vv[u] = q < S.rw.y ? __ldg(v + S.rw.x + q) : (E)0;
        }
    };
    auto fetch_phase = [&](int k, Slot& S) {
        if (k >= ncol) return;
        const int c = back ? ncol - 1 - k : k;
        fetch(s_off[c] + (tid >> 2), s_off[c + 1], S);
    };
    auto phase = [&](int k, Slot& S) {
        const int c = back ? ncol - 1 - k : k, o0 = s_off[c], o1 = s_off[c + 1];
        for (int b0 = o0; b0 < o1; b0 += NT / 4) {
            const int o = b0 + (tid >> 2);
            if (b0 > o0) fetch(o, o1, S);
            E a = (E)0;
#pragma unroll
            for (int u = 0; u < PF; ++u)
                if (sub + 4 * u < S.rw.y) a += S.vv[u] * vec[S.cc[u]];
            for (int q = sub + 4 * PF; q < S.rw.y; q += 4) a += __ldg(v + S.rw.x + q) * vec[__ldg(ci + S.rw.x + q)];
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            if (o < o1) cl_store_every4(&vec[s_beg[c] + o - o0], sub, C, own[o] - a);
        }
        cl_arrive();
        fetch_phase(k + 2, S);
        cl_wait();
    };
    Slot A, B;
    fetch_phase(0, A);
    fetch_phase(1, B);
    for (int k = 0; k < ncol; k += 2) {
        phase(k, A);
        if (k + 1 < ncol) phase(k + 1, B);
    }
}

// FMT 1: skew diagonals; FMT 3: the incomplete factor, J~ = L~^-1 J^ L~^-T.  Its triangular
// solves take one phase per colour (15 to 17 on the 3D stencil, twice per mrs step and twice per
// outer product).  In the launch-by-launch path a phase is a grid barrier after a chain of
// four dependent loads (6 us) or a launch; here a vector being solved for is replicated in the
// shared memory of every CTA, a phase gathers from there, stores its few rows into all CTAs
// and crosses one cluster barrier, with the next colours' entries already on their way: about
// 1 us a phase (mrs steps at 10^3 32 us instead of 129, at 24^3 51 instead of 227).
// GRID: the same solve by one block per SM in a cooperative launch, for systems that a cluster's
// share of the GPU would slow down: a synchronisation is the grid barrier, block sums go through L2
// and every block adds them; what it saves against the launch-by-launch path is the launches and
// the host's part.  A barrier that gives up ends the solve (dead).
// QS (grid scope, FP32): every block keeps its rows of Q_k, more than half of what a row of an mrs
// pass reads, in shared memory for the whole solve, where they fit (at k = 20 up to about 2600
// rows a block, 395 000 in all): 64^3 513 -> 487 us, 70^3 650 -> 596, adjoint at 64^3 543 -> 505,
// 47^3 323 -> 317.  Not in clusters (24^3 249 -> 246, 48^3 with eight columns does not fit), and not
// a part of the rows: the L1 that shared memory takes costs as much (100^3 1423 -> 1425 .. 1481).
// NT: 256 threads where a CTA has few rows, else 512 (see cluster_size).
// WIDE: the FP32 form whose Q_k comes from global memory, for large systems.  Its time hangs on the
// order in which ptxas issues a row's loads, which differs between widths that read the same source: with
// the plain loop over the diagonals a mrs step at 100^3 took 45 us at k = 8 against 35 at k = 20, and at
// 130^3 solves at k = 4, 8 and 12 were slower than launch by launch.  Up to k = 12 the loads of all
// diagonals are issued together (dia_row), and the vectors start on 128 bytes.  Solves at 130^3, k = 4 / 8 /
// 12 / 16 / 20 / 24 / 32, before: 4053 / 5060 / 4015 / 3275 / 3295 / 3631 / 4168 us, now 3117 / 2917 / 3349 / 3295 /
// 3282 / 3340 / 3930; at 100^3 from k = 8 on 1609 / 1454 / 1351 / 1403 / 1519 / 1775, now 1334 / 1449 / 1380 / 1404 /
// 1467 / 1697.  (dia_row at k = 16 / 20 / 24 / 32: 1423 / 1461 / 1532 / 1651.)
template <class T, int KP, int FMT, bool GRID, int NT, bool QS = false>
__global__ void __launch_bounds__(NT, 1) k_solve_cl(const ClArgs<T> p) {
    constexpr int NW = NT / 32, NV = KP + 1, KQ = KP > 0 ? KP : 1;
    using Sh = ClShared<T, KP, GRID, NT>;
    using P2 = typename Sh::P2;
    constexpr bool WIDE = sizeof(T) == 4 && FMT == 1 && GRID && NT == 512 && !QS && KP > 0;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    Sh& sh = *reinterpret_cast<Sh*>(s_dyn);
    double* H = reinterpret_cast<double*>(s_dyn + ((sizeof(Sh) + 15) & ~15));   // (restart + 1) x restart, column-major
    const int R = p.restart, n = p.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = GRID ? (int)blockIdx.x : (int)cl_rank(), C = GRID ? (int)gridDim.x : (int)cl_size();
    const int nsl = (n + 31) >> 5;
    const int rb = (int)((long long)nsl * rank / C) * 32;
    const int re = min(n, (int)((long long)nsl * (rank + 1) / C) * 32);
    const int nact = min(NW, max(re - rb + 31, 0) >> 5);   // warps that hold rows; the others' sums stay zero
    double* base = p.work + (GRID ? (size_t)0 : (size_t)cl_id() * (size_t)p.work_stride);
    const long long nn = WIDE ? pad32(n) : n;
    double *r = base, *rh = r + nn, *t1 = rh + nn, *t2 = t1 + nn, *wv = t2 + nn;
    double* V = wv + nn;
    double* Z = V + (R + 1) * nn;
    T* fb = reinterpret_cast<T*>(Z + R * nn);
    const long long ys = nn + 2LL * p.halo + 32;
    T* Y = fb + p.halo;
    T* P = fb + 3 * ys;
    T* z = P + 2 * nn;

    bool dead = false;      // grid scope: a barrier gave up
    unsigned gphase = p.phase0;
    auto sync_all = [&]() {
        if constexpr (GRID) {
            if (!dead) dead = !grid_sync_phase(p.gb, C, gphase++, p.budget);
        } else {
            cl_sync();
        }
    };
    for (int t = tid; t < p.ndiag && t < 64; t += NT) sh.off[t] = p.off[t];
    if (tid < 64) {
        const ClMat& M = tid < 16 ? p.op1 : tid < 32 ? p.op2 : tid < 48 ? p.Sm : p.Am;
        const int d = tid & 15;
        sh.moff[tid >> 4][d] = d < M.ndiag ? M.off[d] : 0;
    }
    for (int t = tid; t < NW * NV; t += NT) (&sh.wsum[0][0])[t] = (T)0;
    for (int t = tid; t < NW * (CL_REGV + 2); t += NT) (&sh.wd[0][0])[t] = 0.0;
    for (int t = tid; t + 1 < p.k && t < KP; t += NT) sh.alpha[t] = (T)p.alpha[t];
    // the halos of the three Lanczos slots (nothing else writes them)
    for (int t = rank * NT + tid; t < 6 * p.halo; t += C * NT) {
        const int slot = t / (2 * p.halo), e = t % (2 * p.halo);
        Y[slot * ys + (e < p.halo ? e - p.halo : n + (e - p.halo))] = (T)0;
    }
    // FMT 3: replicated vectors, own rows
    const ClFactor<T>& fa = p.fac;
    double* s_vecd = H + (size_t)(R + 1) * R;
    T* s_t = reinterpret_cast<T*>(s_vecd);
    T* s_f = s_t + n;
    double* s_own = nullptr;
    int2 *s_lq = nullptr, *s_uq = nullptr, *s_jq = nullptr;
    int *s_lvl = nullptr, *s_off = nullptr, *s_beg = nullptr;
    if constexpr (FMT == 3) {
        const size_t vb = sizeof(T) == 8 ? 2 * (size_t)n : (size_t)n;   // in doubles
        s_own = s_vecd + vb + (vb & 1);
        s_lq = reinterpret_cast<int2*>(s_own + fa.own_max);
        s_uq = s_lq + fa.own_max;
        s_jq = s_uq + fa.own_max;
        s_lvl = reinterpret_cast<int*>(s_jq + fa.own_max);
        s_off = s_lvl + fa.own_max;
        s_beg = s_off + fa.ncol + 1;
        if (tid == 0) {
            int o = 0;
            for (int c = 0; c < fa.ncol; ++c) {
                const int l0 = fa.ls[c], cnt = fa.ls[c + 1] - l0;
                const int b0 = (int)((long long)cnt * rank / C), b1 = (int)((long long)cnt * (rank + 1) / C);
                s_off[c] = o;
                s_beg[c] = l0 + b0;
                o += b1 - b0;
            }
            s_off[fa.ncol] = o;
        }
        __syncthreads();
        for (int c = 0; c < fa.ncol; ++c)
            for (int o = s_off[c] + tid; o < s_off[c + 1]; o += NT) {
                const int e = s_beg[c] + o - s_off[c];
                s_lvl[o] = fa.lvl[e];
                s_lq[o] = make_int2(fa.L.rp[e], fa.L.rp[e + 1] - fa.L.rp[e]);
                s_uq[o] = make_int2(fa.U.rp[e], fa.U.rp[e + 1] - fa.U.rp[e]);
                s_jq[o] = make_int2(fa.J.rp[e], fa.J.rp[e + 1] - fa.J.rp[e]);
            }
    }
    // own rows of Q_k in shared memory, in the slices of the global copy; on their way until mrs
    float4* s_q = reinterpret_cast<float4*>((reinterpret_cast<size_t>(H + (size_t)(R + 1) * R) + 15) & ~(size_t)15);
    if constexpr (QS) {
        const float4* src = reinterpret_cast<const float4*>(p.Q + (size_t)rb * KP);
        for (int e = tid; e < ((re - rb + 31) >> 5) * 8 * KP; e += NT)
            if (rb + e / (8 * KP) * 32 + (e & 31) < re) cp_async16(s_q + e, src + e);
    }
    sync_all();   // every CTA of the cluster runs: its shared memory may be written

    auto add_t = [](P2 a, P2 b) {
        if constexpr (sizeof(T) == 4) return df_add(a, b);
        else return a + b;
    };
    auto add_d = [](double a, double b) { return a + b; };
    auto now = [&]() -> unsigned long long { return (rank == 0 && tid == 0) ? gtimer() : 0ull; };
    unsigned xphase = 0;
    // out[v] = sum over `rows` rows of a[row * ld + v]: four threads a value
    auto sum_rows = [&](const double* a, int ld, int rows, int cnt, double* out) {
        for (int t0 = 0; t0 < cnt * 4; t0 += NT) {
            const int t = t0 + tid, v = t >> 2;
            double s = 0.0;
            if (v < cnt)
                for (int row = t & 3; row < rows; row += 4) s += a[(size_t)row * ld + v];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (v < cnt && (t & 3) == 0) out[v] = s;
        }
    };
    // cluster totals of the block sums bp[0..cnt) into tot[0..cnt) (a cluster barrier)
    auto exchange = [&](int cnt) {
        __syncthreads();
        const int buf = xphase++ & 1;
        if constexpr (GRID) {
            double* gp = p.part + (size_t)buf * CL_XV * C;
            for (int v = tid; v < cnt; v += NT) gp[(size_t)rank * CL_XV + v] = sh.bp[v];
            sync_all();
            for (int v = warp; v < cnt; v += NW) {   // a warp a value
                double t = 0.0;
                for (int b0 = 0; b0 < C; b0 += 160) {
                    double ld[5];
#pragma unroll
                    for (int u = 0; u < 5; ++u) {
                        const int b = b0 + lane + 32 * u;
                        ld[u] = b < C ? __ldcg(&gp[(size_t)b * CL_XV + v]) : 0.0;
                    }
                    t += (ld[0] + ld[1]) + (ld[2] + ld[3]) + ld[4];
                }
                t = warp_sum(t);
                if (lane == 0) sh.tot[v] = t;
            }
        } else {
            for (int t = tid; t < cnt * C; t += NT) {
                const int q = t / cnt, v = t % cnt;
                cl_store8(&sh.x[buf][rank][v], q, cl_bits(sh.bp[v]));
            }
            sync_all();
            sum_rows(reinterpret_cast<const double*>(&sh.x[buf][0][0]), CL_XV, C, cnt, sh.tot);
        }
        __syncthreads();
    };
    // block sums of CNT accumulators into bp[slot..)
    auto block_sums = [&](auto& acc, int slot) {
        constexpr int CNT = sizeof(acc) / sizeof(double);
        __syncthreads();
        if (warp < nact) warp_fold_to<CNT>(acc, sh.wd[warp]);
        __syncthreads();
        sum_rows(&sh.wd[0][0], CL_REGV + 2, NW, CNT, sh.bp + slot);
    };
    auto norm2 = [&](const double* a) -> double {
        double acc[1] = {0.0};
        for (int i = rb + tid; i < re; i += NT) acc[0] += a[i] * a[i];
        block_sums(acc, 0);
        exchange(1);
        return sh.tot[0];
    };
    // row i of M x (x complete in L2)
    auto mat_row = [&](const ClMat& M, const int* off, const double* x, int i) -> double {
        double s = 0.0;
        if (M.ndiag > 0) {
            for (int d0 = 0; d0 < M.ndiag; d0 += 8) {
                double v[8], xv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int d = d0 + u, j = i + off[d & 15];
                    const bool in = d < M.ndiag && j >= 0 && j < n;
                    const double* vp = &M.val[(size_t)d * n + i];
                    v[u] = in ? (GRID && p.cs ? __ldcs(vp) : __ldg(vp)) : 0.0;
                    xv[u] = in ? x[j] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (d0 + u < M.ndiag) s += v[u] * xv[u];
            }
        } else {
            const int e1 = __ldg(&M.rp[i + 1]);
            for (int e = __ldg(&M.rp[i]); e < e1; e += 8) {
                int cc[8];
                double v[8], xv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    cc[u] = e + u < e1 ? __ldg(&M.ci[e + u]) : 0;
                    v[u] = e + u < e1 ? __ldg(&M.v[e + u]) : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) xv[u] = e + u < e1 ? x[cc[u]] : 0.0;
#pragma unroll
                for (int u = 0; u < 8; ++u) s += v[u] * xv[u];
            }
        }
        return s;
    };

    // out = |D|^-1/2 (I + L)^-1 a, own rows; a complete in L2
    auto apply_F = [&](const double* a, double* out) {
        for (int o = tid; o < s_off[fa.ncol]; o += NT) s_own[o] = a[s_lvl[o]];
        __syncthreads();
        cl_tri_sweep<double, NT>(s_vecd, s_own, s_lq, fa.L.ci, fa.L.d, false, fa.ncol, s_off, s_beg);
        for (int i = rb + tid; i < re; i += NT) {
            double v = fa.wd[i] * s_vecd[fa.pos[i]];
            if (fa.part && fa.part[i] >= 0) v += fa.wo[i] * s_vecd[fa.pos[fa.part[i]]];
            out[i] = v;
        }
    };
    // out = (I + L)^-T |D|^-1/2 a, own rows; a complete in L2
    auto apply_G = [&](const double* a, double* out) {
        for (int o = tid; o < s_off[fa.ncol]; o += NT) {
            const int i = s_lvl[o];
            double v = fa.wd[i] * a[i];
            if (fa.part && fa.part[i] >= 0) v += fa.wo[i] * a[fa.part[i]];
            s_own[o] = v;
        }
        __syncthreads();
        cl_tri_sweep<double, NT>(s_vecd, s_own, s_uq, fa.U.ci, fa.U.d, true, fa.ncol, s_off, s_beg);
        for (int i = rb + tid; i < re; i += NT) out[i] = s_vecd[fa.pos[i]];
    };
    // s_f = (I + L)^-1 J^ (I + L)^-T (wd .* y) by position, y complete in L2
    auto apply_skew = [&](const T* y) {
        T* own = reinterpret_cast<T*>(s_own);
        for (int o = tid; o < s_off[fa.ncol]; o += NT) {
            const int i = s_lvl[o];
            T v = __ldg(&fa.wdT[i]) * y[i];
            if (fa.part && __ldg(&fa.part[i]) >= 0) v += __ldg(&fa.woT[i]) * y[__ldg(&fa.part[i])];
            own[o] = v;
        }
        __syncthreads();
        cl_tri_sweep<T, NT>(s_t, own, s_uq, fa.U.ci, fa.U.v, true, fa.ncol, s_off, s_beg);
        for (int o = tid; o < s_off[fa.ncol]; o += NT) {
            const int2 rw = s_jq[o];
            T a = (T)0;
            for (int q = 0; q < rw.y; q += 12) {
                int cc[12];
                T vv[12];
#pragma unroll
                for (int u = 0; u < 12; ++u) {
                    cc[u] = q + u < rw.y ? __ldg(fa.J.ci + rw.x + q + u) : 0;
                    vv[u] = q + u < rw.y ? __ldg(fa.J.v + rw.x + q + u) : (T)0;
                }
#pragma unroll
                for (int u = 0; u < 12; ++u)
                    if (q + u < rw.y) a += vv[u] * s_t[cc[u]];
            }
            own[o] = a;
        }
        __syncthreads();
        cl_tri_sweep<T, NT>(s_f, own, s_lq, fa.L.ci, fa.L.v, false, fa.ncol, s_off, s_beg);
    };

    // ---------------------------------------------------------------------------
    // mrs (App. B) on (I + sign (J~ - Q S_k Q^T)) z = u; Q^T z into sh.wv[0..k)
    // ---------------------------------------------------------------------------
    auto mrs_sums = [&](T(&tacc)[NV]) {   // cluster totals into sh.red, for warp 0
        if (warp < nact) warp_fold_to<NV>(tacc, sh.wsum[warp]);
        __syncthreads();
        const int buf = xphase++ & 1;
        if (warp == 0) {
            for (int v = lane; v < NV; v += 32) {
                P2 a[NW];
#pragma unroll
                for (int q = 0; q < NW; ++q) {
                    if constexpr (sizeof(T) == 4) a[q] = make_float2(sh.wsum[q][v], 0.f);
                    else a[q] = sh.wsum[q][v];
                }
                const unsigned long long bits = cl_bits(pair_tree(a, add_t));
                if constexpr (GRID)
                    reinterpret_cast<unsigned long long*>(p.part + (size_t)buf * CL_XV * C)[(size_t)rank * NV + v] = bits;
                else
                    for (int q = 0; q < C; ++q) cl_store8(&sh.x[buf][rank][v], q, bits);
            }
        }
        sync_all();
        if constexpr (GRID) {
            // as k_mrs: FP32 a warp every 16th block, a lane a value; FP64 a lane an addition
            const P2* gp = reinterpret_cast<const P2*>(p.part + (size_t)buf * CL_XV * C);
            P2* bs = reinterpret_cast<P2*>(&sh.bsum[0][0]);
            constexpr int NG = sizeof(T) == 4 ? NW : NT / NV, UB = NT == 256 ? 20 : 10;   // UB: parts in flight
            for (int t = tid; t < (sizeof(T) == 4 ? NT : NG * NV); t += NT) {
                const int g = sizeof(T) == 4 ? warp : t / NV;
                for (int v = sizeof(T) == 4 ? lane : t % NV; v < NV; v += sizeof(T) == 4 ? 32 : NV) {
                    P2 acc{};
                    for (int b0 = g; b0 < C; b0 += NG * UB) {
                        P2 ld[UB];
#pragma unroll
                        for (int u = 0; u < UB; ++u) {
                            const int b = b0 + u * NG;
                            ld[u] = b < C ? __ldcg(&gp[(size_t)b * NV + v]) : P2{};
                        }
#pragma unroll
                        for (int u = 0; u < UB; ++u)
                            if (b0 + u * NG < C) acc = add_t(acc, ld[u]);
                    }
                    bs[g * NV + v] = acc;
                }
            }
            __syncthreads();
            if constexpr (sizeof(T) == 4) {
                if (warp == 0) {
                    for (int v = lane; v < NV; v += 32) {
                        P2 a[NW];
#pragma unroll
                        for (int q = 0; q < NW; ++q) a[q] = bs[q * NV + v];
                        const P2 t = pair_tree(a, add_t);
                        sh.red[v] = t.x + t.y;
                    }
                    __syncwarp();
                }
            } else {
                for (int t0 = 0; t0 < 4 * NV; t0 += NT) {
                    const int t = t0 + tid, v = t >> 2;
                    double a = 0.0;
                    if (v < NV)
                        for (int g = t & 3; g < NG && g < C; g += 4) a += sh.bsum[g][v];
                    a += __shfl_xor_sync(0xffffffffu, a, 1);
                    a += __shfl_xor_sync(0xffffffffu, a, 2);
                    if (v < NV && (t & 3) == 0) sh.red[v] = (T)a;
                }
                __syncthreads();
            }
        } else if (warp == 0) {
            for (int v = lane; v < NV; v += 32) {
                P2 a[CL_MAX];
#pragma unroll
                for (int q = 0; q < CL_MAX; ++q) {
                    a[q] = P2{};
                    if (q < C) a[q] = *reinterpret_cast<const P2*>(&sh.x[buf][q][v]);
                }
                const P2 t = pair_tree(a, add_t);
                if constexpr (sizeof(T) == 4) sh.red[v] = t.x + t.y;
                else sh.red[v] = t;
            }
            __syncwarp();
        }
    };
    auto make_u = [&]() {   // u = S_k (nu Q^T y), warp 0
        for (int a = lane; a < KP; a += 32) {
            T u = (T)0;
            if (a < p.k) {
                if (a + 1 < p.k) u += sh.alpha[a] * sh.red[2 + a] * sh.sc.nu;
                if (a > 0) u -= sh.alpha[a - 1] * sh.red[a] * sh.sc.nu;
            }
            sh.u[a] = u;
        }
    };
    auto set_coefs = [&]() {
        const MrsScalars<T>& c = sh.sc;
        sh.cf[0] = (T)p.sign * c.nu;
        sh.cf[1] = (T)p.sign;
        sh.cf[2] = c.coef_old;
        sh.cf[3] = c.nu_p;
        sh.cf[4] = c.delta_pp;
        sh.cf[5] = c.rtheta_p;
        sh.cf[6] = c.xcoef_p;
        if (c.stop) {
            sh.cf[7] = c.fin_nu;
            sh.cf[8] = c.fin_delta;
            sh.cf[9] = c.fin_rtheta;
            sh.cf[10] = c.fin_xcoef;
        }
    };
    auto qtx_fold = [&](int jj) {   // warp 1: direction p_jj into Q^T z
        for (int a = lane; a < p.k; a += 32) {
            T* pp = sh.qtp[jj & 1];
            const T v = (sh.pq[0] * sh.qty[a] - sh.pq[1] * pp[a]) * sh.pq[2];
            pp[a] = v;
            sh.qtx[a] += sh.pq[3] * v;
        }
    };
    auto mrs = [&](const double* rhs) -> int {
        for (int a = tid; a < KP; a += NT) {
            sh.qtp[0][a] = (T)0;
            sh.qtp[1][a] = (T)0;
            sh.qtx[a] = (T)0;
        }
        if constexpr (QS) {
            cp_async_wait_all();
            __syncthreads();
        }
        T tacc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) tacc[v] = (T)0;
        for (int i = rb + tid; i < re; i += NT) {
            const T b = (T)rhs[i];
            Y[i] = b;
            z[i] = (T)0;
            P[i] = (T)0;
            P[nn + i] = (T)0;
            tacc[0] += b * b;
            T q[KQ];
            cl_qrow<T, KP, QS>(p.Q, s_q, rb, i, q, GRID && p.cs);
#pragma unroll
            for (int a = 0; a < KP; ++a) tacc[1 + a] += q[a] * b;
        }
        mrs_sums(tacc);
        if (GRID && dead) return 0;
        if (warp == 0) {
            if (lane == 0) {
                MrsScalars<T>& c = sh.sc;
                const T r0 = sqrt(sh.red[0]);
                c.r0 = r0;
                c.rr0 = r0 > (T)0 ? (T)1 / r0 : (T)0;
                c.nu = c.rr0;
                c.coef_old = (T)0;
                c.theta_t = (T)1;
                c.c_prev = (T)1;
                c.s_prev = (T)0;
                c.delta_prev = (T)0;
                c.G = r0;
                c.nu_p = (T)0;
                c.delta_pp = (T)0;
                c.rtheta_p = (T)1;
                c.xcoef_p = (T)0;
                c.its = 0;
                c.stop = r0 > (T)0 ? 0 : 1;
                set_coefs();
            }
            __syncwarp();
            if (!sh.sc.stop) make_u();
        }
        __syncthreads();
        if (sh.sc.stop) {
            for (int a = tid; a < p.k; a += NT) sh.wv[a] = (T)0;
            return 0;
        }
        for (int j = 1; j <= p.inner_maxit; ++j) {
            if (KP > 0 && warp == 1) {
                if (j >= 2) qtx_fold(j - 1);
                for (int a = lane; a < p.k; a += 32) sh.qty[a] = sh.red[1 + a];
            }
            const T* Ycur = Y + (size_t)((j - 1) % 3) * ys;
            const T* __restrict__ Yold = Y + (size_t)((j + 1) % 3) * ys;   // own rows
            T* __restrict__ Ynew = Y + (size_t)(j % 3) * ys;
            T* __restrict__ Pj1 = P + (size_t)((j - 1) & 1) * nn;
            T* __restrict__ zz = z;
            const T tnu = sh.cf[0], tsg = sh.cf[1], tco = sh.cf[2], tnp = sh.cf[3], tdpp = sh.cf[4], tthp = sh.cf[5],
                    txp = sh.cf[6];
#pragma unroll
            for (int v = 0; v < NV; ++v) tacc[v] = (T)0;
            if constexpr (FMT == 3) apply_skew(Ycur);
            for (int i = rb + tid; i < re; i += NT) {
                const T yold = j >= 2 ? Yold[i] : (T)0;
                const T pold = j >= 2 ? Pj1[i] : (T)0;
                // with the first loads, as in k_mrs (100^3: 1439 -> 1423 us a solve, 47^3 326 -> 319)
                const T zold = j >= 2 ? zz[i] : (T)0;
                T acc = (T)0;
                if constexpr (FMT == 3) {
                    acc = __ldg(&fa.wdT[i]) * s_f[__ldg(&fa.pos[i])];
                    if (fa.part && __ldg(&fa.part[i]) >= 0)
                        acc += __ldg(&fa.woT[i]) * s_f[__ldg(&fa.pos[__ldg(&fa.part[i])])];
                }
                const T* Ud = p.U + i;
                const T* yi = Ycur + i;
                if constexpr (WIDE && KP <= 12) {
                    acc = dia_row<T, 12>(Ud, p.ustride, yi, sh.off, p.ndiag);
                } else {
#pragma unroll 12
                    for (int d = 0; d < (FMT == 1 ? p.ndiag : 0); ++d, Ud += p.ustride) {
                        const int mo = sh.off[d];
                        if constexpr (sizeof(T) == 8) {
                            acc = fma(__ldg(Ud), yi[mo], acc);
                            acc = fma(-__ldg(Ud - mo), yi[-mo], acc);
                        } else {
                            acc += __ldg(Ud) * yi[mo] - __ldg(Ud - mo) * yi[-mo];
                        }
                    }
                }
                T q[KQ];
                cl_qrow<T, KP, QS>(p.Q, s_q, rb, i, q, GRID && p.cs);
                T dq = (T)0;
#pragma unroll
                for (int a = 0; a < KP; ++a) dq += q[a] * sh.u[a];
                const T ynew = tnu * acc - tsg * dq + tco * yold;
                Ynew[i] = ynew;
                tacc[0] += ynew * ynew;
#pragma unroll
                for (int a = 0; a < KP; ++a) tacc[1 + a] += q[a] * ynew;
                if (j >= 2) {
                    const T pv = (tnp * yold - tdpp * pold) * tthp;
                    Pj1[i] = pv;
                    zz[i] = zold + txp * pv;
                }
            }
            mrs_sums(tacc);
            if (GRID && dead) break;
            if (warp == 0) {
                MrsScalars<T>& c = sh.sc;
                // beta and 1 / beta in lane 0, theta and 1 / theta in lane 1
                const T rad = lane == 0 ? sh.red[0] : c.theta_t * c.theta_t + sh.red[0];
                T root, inv;
                if constexpr (sizeof(T) == 4) {
                    root = sqrt(rad);
                    inv = (T)1 / root;
                } else {
                    inv = rsqrt(rad);
                    root = rad != (T)0 ? rad * inv : (T)0;
                }
                const T beta = __shfl_sync(0xffffffffu, root, 0), rbeta = __shfl_sync(0xffffffffu, inv, 0);
                const T theta = __shfl_sync(0xffffffffu, root, 1), rth = __shfl_sync(0xffffffffu, inv, 1);
                if (lane == 0) {
                    const T cc = c.theta_t * rth, s = beta * rth;
                    const T delta = -c.s_prev * beta;
                    const T theta_t_next = c.c_prev * theta;
                    const T xcoef = c.G * cc;
                    const T Gn = -c.G * s;
                    sh.pq[0] = c.nu;
                    sh.pq[1] = c.delta_prev;
                    sh.pq[2] = rth;
                    sh.pq[3] = xcoef;
                    c.ratio = fabs(Gn) * c.rr0;
                    c.its = j;
                    if (c.ratio < (T)p.inner_tol || j == p.inner_maxit) {
                        c.stop = 1;
                        c.fin_nu = c.nu;
                        c.fin_delta = c.delta_prev;
                        c.fin_rtheta = rth;
                        c.fin_xcoef = xcoef;
                    } else {
                        c.nu_p = c.nu;
                        c.delta_pp = c.delta_prev;
                        c.rtheta_p = rth;
                        c.xcoef_p = xcoef;
                        c.coef_old = beta * c.nu;
                        c.nu = (beta != (T)0) ? rbeta : (T)0;
                        c.s_prev = s;
                        c.c_prev = cc;
                        c.delta_prev = delta;
                        c.theta_t = theta_t_next;
                        c.G = Gn;
                    }
                    set_coefs();
                }
                __syncwarp();
                if (!sh.sc.stop) make_u();
            }
            __syncthreads();
            if (sh.sc.stop) {
                const T* Pj = P + (size_t)(j & 1) * nn;
                const T tn = sh.cf[7], td = sh.cf[8], tth = sh.cf[9], tx = sh.cf[10];
                for (int i = rb + tid; i < re; i += NT) {
                    const T pv = (tn * Ycur[i] - td * Pj[i]) * tth;
                    z[i] = z[i] + tx * pv;
                }
                if (KP > 0 && warp == 1) {
                    qtx_fold(j);
                    __syncwarp();
                    for (int a = lane; a < p.k; a += 32) sh.wv[a] = sh.qtx[a];
                }
                break;
            }
        }
        return sh.sc.its;
    };

    // f(count as a constant) for the vector counts whose dot products run together
    auto by_count = [&](int nv, auto f) {
        switch (nv) {
            case 1: f(std::integral_constant<int, 1>{}); break;
            case 2: f(std::integral_constant<int, 2>{}); break;
            case 3: f(std::integral_constant<int, 3>{}); break;
            case 4: f(std::integral_constant<int, 4>{}); break;
            case 5: f(std::integral_constant<int, 5>{}); break;
            default: f(std::integral_constant<int, 6>{}); break;
        }
    };
    // block sums of V_a^T w, a < nv, one warp per vector, into bp[0..nv)
    auto dots_by_warp = [&](int nv) {
        __syncthreads();
        for (int a = warp; a < nv; a += NW) {
            const double* va = V + (size_t)a * nn;
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            int i = rb + lane;
            for (; i + 96 < re; i += 128)
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] += va[i + u * 32] * wv[i + u * 32];
            for (; i < re; i += 32) acc[0] += va[i] * wv[i];
            const double t = warp_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
            if (lane == 0) sh.bp[a] = t;
        }
    };
    auto project = [&](int i, int nv, const double* h) -> double {
        double s = 0.0;
        for (int a = 0; a < nv; a += 8) {
            double ld[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) ld[u] = a + u < nv ? V[(size_t)(a + u) * nn + i] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (a + u < nv) s += ld[u] * h[a + u];
        }
        return wv[i] - s;
    };

    for (int col = GRID ? 0 : (int)cl_id(); col < p.ncol; col += GRID ? 1 : (int)cl_count()) {
        const double* b = p.b + (size_t)col * p.ldb;
        double* x = p.x + (size_t)col * p.ldx;
        unsigned long long ns_inner = 0, ns_op = 0, ns_orth = 0;
        int outer = 0, cycles = 0, status = ASSS_OK, stall = 0, solves = 0, ops = 0, orths = 0;
        long long inner = 0, vecs = 0;
        double relres = 0.0, best = INFINITY;
        for (int i = rb + tid; i < re; i += NT) {
            x[i] = 0.0;
            r[i] = b[i];
        }
        const double bn = sqrt(norm2(r));
        double rn = bn;
        if (!(bn < INFINITY)) {   // a NaN or an infinity in b
            status = ASSS_ERR_BREAKDOWN;
            relres = 1.0;
        }
        if (GRID && dead) status = ASSS_ERR_TIMEOUT;
        // a right-hand side of norm 0, infinity or NaN counts the one inner solve of zero steps
        // that the launch-by-launch path has enqueued by the time it knows
        if (!(bn > 0.0 && bn < INFINITY) && p.outer_tol < 1.0 && p.outer_maxit > 0) solves = 1;
        while (bn > 0.0 && status == ASSS_OK) {
            relres = rn / bn;
            if (relres <= p.outer_tol) break;
            if (!(rn == rn)) {
                status = ASSS_ERR_BREAKDOWN;
                break;
            }
            if (outer >= p.outer_maxit) {
                status = ASSS_ERR_NOT_CONVERGED;
                break;
            }
            if (rn < 0.999 * best) {
                best = rn;
                stall = 0;
            } else if (++stall >= 5) {
                status = ASSS_ERR_STAGNATION;
                break;
            }
            // r^ = W P D_r r, or W S^T D_c r (the barrier of the last norm published r)
            // (FMT 3: F P D_r r or F S^T D_c r, W = 1 there)
            double* rs = FMT == 3 ? t2 : rh;
            if (!p.tr) {
                for (int i = rb + tid; i < re; i += NT) {
                    const int q = p.perm ? p.perm[i] : i;
                    rs[i] = p.w[i] * p.dr[q] * r[q];
                }
            } else {
                for (int i = rb + tid; i < re; i += NT) t1[i] = p.dc[i] * r[i];
                sync_all();
                for (int i = rb + tid; i < re; i += NT) rs[i] = p.w[i] * mat_row(p.Sm, sh.moff[2], t1, i);
            }
            if constexpr (FMT == 3) {
                sync_all();
                apply_F(rs, rh);
            }
            const double eta = fmin(0.5, 0.5 * p.outer_tol * bn / rn);
            const int mcyc = min(R, p.outer_maxit - outer);
            // ---- one flexible GMRES cycle ----
            const double rr = norm2(rh);
            int steps = 0;
            if (rr > 0.0 && rr < INFINITY) {
                const double beta0 = sqrt(rr), inv0 = 1.0 / beta0, thr = eta * beta0;
                for (int i = rb + tid; i < re; i += NT) V[i] = inv0 * rh[i];
                if (tid == 0) sh.g[0] = beta0;
                for (int j = 0; j < mcyc; ++j) {
                    double* zj = Z + (size_t)j * nn;
                    const unsigned long long tm0 = now();
                    inner += mrs(V + (size_t)j * nn);
                    const unsigned long long tm1 = now();
                    ++solves;
                    // z_j = z - Y (U^T z)
                    if (p.r > 0 && p.m > 0) {
                        sync_all();   // z complete: U_r^T z gathers from every CTA's rows
                        for (int a = tid; a < p.r; a += NT) {
                            double v;
                            if (!p.neg2) {
                                v = (double)z[p.neg[a]];
                            } else {
                                v = p.negc1[a] * (double)z[p.neg[a]];
                                const int q = p.neg2[a];
                                if (q >= 0) v += p.negc2[a] * (double)z[q];
                            }
                            sh.wv[p.k + a] = (T)v;
                        }
                    }
                    __syncthreads();
                    for (int i = rb + tid; i < re; i += NT) {
                        T acc = (T)0;
                        const T* yr = p.Ys + (size_t)i * p.m;
                        if (sizeof(T) == 4 && (p.m & 3) == 0) {
                            const float4* y4 = reinterpret_cast<const float4*>(yr);
#pragma unroll 5
                            for (int c = 0; c < (p.m >> 2); ++c) {
                                const float4 v = GRID && p.cs ? __ldcs(y4 + c) : __ldg(y4 + c);
                                acc += (T)v.x * sh.wv[4 * c] + (T)v.y * sh.wv[4 * c + 1] + (T)v.z * sh.wv[4 * c + 2] +
                                       (T)v.w * sh.wv[4 * c + 3];
                            }
                        } else {
                            for (int c = 0; c < p.m; ++c) acc += yr[c] * sh.wv[c];
                        }
                        zj[i] = (double)(z[i] - acc);
                    }
                    // w = A_cal z_j
                    sync_all();
                    const unsigned long long tm2 = now();
                    if constexpr (FMT == 3) {   // F A^ G z_j
                        apply_G(zj, t2);
                        sync_all();
                    }
                    const double* zin = FMT == 3 ? t2 : zj;
                    for (int i = rb + tid; i < re; i += NT) t1[i] = mat_row(p.op1, sh.moff[0], zin, i);
                    sync_all();
                    double* wout = FMT == 3 ? t2 : wv;
                    for (int i = rb + tid; i < re; i += NT) wout[i] = mat_row(p.op2, sh.moff[1], t1, i);
                    if constexpr (FMT == 3) {
                        sync_all();
                        apply_F(t2, wv);
                    }
                    const unsigned long long tm3 = now();
                    ++ops;
                    // two classical Gram-Schmidt passes; ||w2||^2 = ||w1||^2 - ||h2||^2
                    const int nv = j + 1;
                    vecs += nv;
                    if (nv <= CL_REGV) {
                        by_count(nv, [&](auto nvc) {
                            constexpr int NVC = decltype(nvc)::value;
                            double acc[NVC];
#pragma unroll
                            for (int t = 0; t < NVC; ++t) acc[t] = 0.0;
                            for (int i = rb + tid; i < re; i += NT) {
                                const double wi = wv[i];
#pragma unroll
                                for (int t = 0; t < NVC; ++t) acc[t] += V[(size_t)t * nn + i] * wi;
                            }
                            block_sums(acc, 0);
                        });
                    } else {
                        dots_by_warp(nv);
                    }
                    exchange(nv);
                    for (int a = tid; a < nv; a += NT) sh.h1[a] = sh.tot[a];
                    if (nv <= CL_REGV) {
                        by_count(nv, [&](auto nvc) {
                            constexpr int NVC = decltype(nvc)::value;
                            double acc[NVC + 1], h[NVC];
#pragma unroll
                            for (int t = 0; t <= NVC; ++t) acc[t] = 0.0;
#pragma unroll
                            for (int t = 0; t < NVC; ++t) h[t] = sh.tot[t];
                            for (int i = rb + tid; i < re; i += NT) {
                                double vi[NVC], s = 0.0;
#pragma unroll
                                for (int t = 0; t < NVC; ++t) {
                                    vi[t] = V[(size_t)t * nn + i];
                                    s += vi[t] * h[t];
                                }
                                const double wn = wv[i] - s;
                                wv[i] = wn;
#pragma unroll
                                for (int t = 0; t < NVC; ++t) acc[t] += vi[t] * wn;
                                acc[NVC] += wn * wn;
                            }
                            block_sums(acc, 0);
                        });
                    } else {
                        double acc[1] = {0.0};
                        for (int i = rb + tid; i < re; i += NT) {
                            const double wn = project(i, nv, sh.tot);
                            wv[i] = wn;
                            acc[0] += wn * wn;
                        }
                        block_sums(acc, nv);
                        dots_by_warp(nv);
                    }
                    exchange(nv + 1);
                    if (warp == 0) {   // the norm, then the Givens update (every CTA the same)
                        double h2n = 0.0;
                        for (int a = 0; a < nv; ++a) h2n += sh.tot[a] * sh.tot[a];
                        const double hn2 = fmax(sh.tot[nv] - h2n, 0.0);
                        const double inv = hn2 > 0.0 ? rsqrt(hn2) : 0.0, hn = hn2 * inv;
                        if (lane == 0) {
                            sh.fin[0] = hn2;
                            sh.fin[1] = hn;
                            sh.fin[2] = inv;
                        }
                    }
                    __syncthreads();
                    const double inv = sh.fin[2];
                    double* vn = V + (size_t)nv * nn;
                    for (int i = rb + tid; i < re; i += NT) vn[i] = project(i, nv, sh.tot) * inv;
                    if (tid == NT - 1) {
                        const double hn2 = sh.fin[0], hn = sh.fin[1];
                        double* hc = H + (size_t)j * (R + 1);
                        double cur = sh.h1[0] + sh.tot[0];
                        for (int a = 0; a < j; ++a) {
                            const double next = sh.h1[a + 1] + sh.tot[a + 1];
                            hc[a] = sh.cs[a] * cur + sh.sn[a] * next;
                            cur = sh.cs[a] * next - sh.sn[a] * cur;
                        }
                        const double big = fmax(fabs(cur), hn);
                        double rot, c, s;
                        if (big > 1e-140 && big < 1e140) {
                            const double q2 = cur * cur + hn * hn, ir = rsqrt(q2);
                            rot = q2 * ir;
                            c = cur * ir;
                            s = hn * ir;
                        } else {
                            rot = hypot(cur, hn);
                            c = (rot != 0.0) ? cur / rot : 1.0;
                            s = (rot != 0.0) ? hn / rot : 0.0;
                        }
                        hc[j] = rot;
                        sh.cs[j] = c;
                        sh.sn[j] = s;
                        const double gj = sh.g[j];
                        sh.g[j + 1] = -s * gj;
                        sh.g[j] = c * gj;
                        sh.stop = (hn2 == 0.0 || fabs(s * gj) <= thr) ? 1 : 0;
                    }
                    __syncthreads();
                    const unsigned long long tm4 = now();
                    ns_inner += tm1 - tm0;
                    ns_op += tm3 - tm2;
                    ns_orth += tm4 - tm3;
                    ++orths;
                    steps = j + 1;
                    if (sh.stop || (GRID && dead)) break;
                }
                // y from the triangular system, column by column
                if (warp == 0) {
                    for (int a = lane; a < steps; a += 32) sh.yv[a] = sh.g[a];
                    __syncwarp();
                    for (int a = steps - 1; a >= 0; --a) {
                        const double ya = sh.yv[a] / H[(size_t)a * (R + 1) + a];
                        __syncwarp();
                        for (int q = lane; q < a; q += 32) sh.yv[q] -= H[(size_t)a * (R + 1) + q] * ya;
                        if (lane == 0) sh.yv[a] = ya;
                        __syncwarp();
                    }
                }
                __syncthreads();
            }
            // x += D_c S W dy, or lambda += D_r P^T W dy, with dy = Z y
            for (int i = rb + tid; i < re; i += NT) {
                double dy = 0.0;
                for (int a = 0; a < steps; a += 8) {
                    double ld[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) ld[u] = a + u < steps ? Z[(size_t)(a + u) * nn + i] : 0.0;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (a + u < steps) dy += ld[u] * sh.yv[a + u];
                }
                if (FMT == 3) {
                    t2[i] = dy;
                } else if (!p.tr) {
                    t1[i] = p.w[i] * dy;
                } else {
                    const int q = p.perm ? p.perm[i] : i;
                    x[q] += p.dr[q] * p.w[i] * dy;
                }
            }
            sync_all();
            if constexpr (FMT == 3) {   // G dy instead of W dy
                apply_G(t2, t1);
                if (p.tr)
                    for (int i = rb + tid; i < re; i += NT) {
                        const int q = p.perm ? p.perm[i] : i;
                        x[q] += p.dr[q] * t1[i];
                    }
                sync_all();
            }
            if (!p.tr) {
                for (int i = rb + tid; i < re; i += NT) x[i] += p.dc[i] * mat_row(p.Sm, sh.moff[2], t1, i);
                sync_all();
            }
            for (int i = rb + tid; i < re; i += NT) r[i] = b[i] - mat_row(p.Am, sh.moff[3], x, i);
            outer += steps;
            ++cycles;
            rn = sqrt(norm2(r));
            if (GRID && dead) status = ASSS_ERR_TIMEOUT;
        }
        if (rank == 0 && tid == 0) {
            ClStat st;
            st.outer_its = outer;
            st.cycles = cycles;
            st.status = status;
            st.solves = solves;
            st.op_calls = ops;
            st.orth_calls = orths;
            st.inner_its = inner;
            st.orth_vecs = vecs;
            st.ns_inner = ns_inner;
            st.ns_op = ns_op;
            st.ns_orth = ns_orth;
            st.relres = relres;
            st.phase = gphase + 1;   // with the column's last barrier, below
            p.stats[col] = st;
        }
        sync_all();   // the column is done before its buffers are reused
        if (GRID && dead) return;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// clusters of `size` CTAs that can be resident at once (0: none fits)
template <class T, int KP, int FMT, int NT>
static asss_status cl_clusters(int size, size_t smem, int* count) {
    const void* fn = (const void*)k_solve_cl<T, KP, FMT, false, NT>;
    ASSS_TRY(raise_dynamic_smem(fn, (int)smem));
    if (size > 8) ASSS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = size;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(count, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();   // a size this device does not take
        *count = 0;
    }
    return ASSS_OK;
}

// launches `count` clusters of `size` CTAs, or (size == 0) asks how many clusters of each of
// CL_SIZES can be resident, into counts
template <class T, int KP, int FMT, int NT>
static asss_status cl_run(const Ctx& c, const ClArgs<T>& a, int size, int count, int* counts) {
    ClArgs<T> b = a;
    auto bytes = [&](int sz) -> size_t {
        size_t smem = ((sizeof(ClShared<T, KP, false, NT>) + 15) & ~(size_t)15) +
                      sizeof(double) * (size_t)(a.restart + 1) * (size_t)a.restart;
        if (FMT == 3) {
            b.fac.own_max = a.n / sz + a.fac.ncol + 1;
            smem += (size_t)cl_factor_smem<T>(a.n, b.fac.own_max, a.fac.ncol);
        }
        return smem;
    };
    if (size == 0) {
        for (int t = 0; t < CL_NSIZES; ++t) {
            const size_t need = bytes(CL_SIZES[t]);
            counts[t] = 0;
            if (need <= CL_SMEM_MAX) ASSS_TRY((cl_clusters<T, KP, FMT, NT>(CL_SIZES[t], need, &counts[t])));
        }
        return ASSS_OK;
    }
    const size_t smem = bytes(size);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size * count);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = size;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ASSS_CUDA(cudaLaunchKernelEx(&cfg, k_solve_cl<T, KP, FMT, false, NT>, b));
    count_launch();
    return ASSS_OK;
}

// grid scope: a cooperative launch of one block per SM (size < 0)
template <class T, int KP, int NT>
static asss_status cl_run_grid(const Ctx& c, const ClArgs<T>& a) {
    size_t smem = ((sizeof(ClShared<T, KP, true, NT>) + 15) & ~(size_t)15) +
                  sizeof(double) * (size_t)(a.restart + 1) * (size_t)a.restart;
    const int need = cdiv(a.n, 32), blocks = c.sms < need ? c.sms : need;
    const size_t q = sizeof(T) == 4 && KP > 0 ? cl_q_bytes(a.n, KP, blocks, smem) : 0;
    const void* fn = nullptr;
    if constexpr (sizeof(T) == 4 && KP > 0) {
        if (q) fn = (const void*)k_solve_cl<T, KP, 1, true, NT, true>;
    }
    if constexpr (sizeof(T) == 8 || NT == 512) {
        if (!q) fn = (const void*)k_solve_cl<T, KP, 1, true, NT>;
    }
    if (!fn) {   // (few rows a block: they fit)
        set_error("solve: Q_k does not fit shared memory");
        return ASSS_ERR_UNSUPPORTED;
    }
    smem += q;
    ClArgs<T> b = a;
    ASSS_TRY(raise_dynamic_smem(fn, (int)smem));
    void* args[] = {&b};
    ASSS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(NT), args, smem, c.stream));
    count_launch();
    return ASSS_OK;
}

// (FP64 on diagonals takes 512 threads in grid scope only)
template <class T, int FMT, int NT>
asss_status cl_dispatch(const Ctx& c, const ClArgs<T>& a, int kp, int size, int count, int* counts) {
    constexpr bool CLUSTERS = !(sizeof(T) == 8 && FMT == 1 && NT == 512);
    switch (kp) {
#define ASSS_CL_CASE(KPV) \
    case KPV:             \
        if constexpr (FMT == 1) { if (size < 0) return cl_run_grid<T, KPV, NT>(c, a); } \
        if constexpr (CLUSTERS) return cl_run<T, KPV, FMT, NT>(c, a, size, count, counts); \
        break;
        ASSS_CL_CASE(4)
        ASSS_CL_CASE(8)
        ASSS_CL_CASE(12)
        ASSS_CL_CASE(16)
        ASSS_CL_CASE(20)
        ASSS_CL_CASE(24)
        ASSS_CL_CASE(32)
        case 0:
            if constexpr (sizeof(T) == 8 || NT == 512) {
                if constexpr (FMT == 1) { if (size < 0) return cl_run_grid<T, 0, NT>(c, a); }
                if constexpr (CLUSTERS) return cl_run<T, 0, FMT, NT>(c, a, size, count, counts);
            }
            break;
#undef ASSS_CL_CASE
    }
    set_error("cluster solve: unsupported padded Lanczos width %d", kp);
    return ASSS_ERR_UNSUPPORTED;
}

// (solve_cluster32.cu, solve_cluster32s.cu, solve_cluster64.cu, solve_cluster64w.cu, solve_cluster_fac32.cu,
// solve_cluster_fac64.cu)
extern template asss_status cl_dispatch<float, 1, 512>(const Ctx&, const ClArgs<float>&, int, int, int, int*);
extern template asss_status cl_dispatch<float, 1, 256>(const Ctx&, const ClArgs<float>&, int, int, int, int*);
extern template asss_status cl_dispatch<double, 1, 512>(const Ctx&, const ClArgs<double>&, int, int, int, int*);
extern template asss_status cl_dispatch<double, 1, 256>(const Ctx&, const ClArgs<double>&, int, int, int, int*);
extern template asss_status cl_dispatch<float, 3, 512>(const Ctx&, const ClArgs<float>&, int, int, int, int*);
extern template asss_status cl_dispatch<double, 3, 512>(const Ctx&, const ClArgs<double>&, int, int, int, int*);

}  // namespace asss
