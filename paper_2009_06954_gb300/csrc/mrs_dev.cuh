// Device helpers shared by the single- and multi-right-hand-side mrs kernels.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace asss {

constexpr int MRS_THREADS = 512;
constexpr int MRS_WARPS = MRS_THREADS / 32;
constexpr int MRS_KPMAX = 64;
constexpr int MRS_MAXDIAG = 64;

// BF16 rows: KP a multiple of 8, 16-byte aligned, converted to T on load
template <class T, int KP>
__device__ __forceinline__ void load_qrow16(const __nv_bfloat16* __restrict__ Q, int i, T (&q)[KP > 0 ? KP : 1]) {
    if constexpr (KP > 0) {
        const __nv_bfloat16* row = Q + (size_t)i * KP;
#pragma unroll
        for (int m = 0; m < KP; m += 8) {
            uint4 v = *reinterpret_cast<const uint4*>(row + m);
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                float2 f = __bfloat1622float2(h[t]);
                q[m + 2 * t] = (T)f.x;
                q[m + 2 * t + 1] = (T)f.y;
            }
        }
    }
}

// Whether Q_k is stored in slices of 32 rows (FP32, operators that visit the rows in their
// natural order: natural = true) or row by row.  In a slice the four values m..m+3 of
// its 32 rows stand side by side, so a warp's load is 512 contiguous bytes; the same load
// of 80-byte rows touched 20 lines, five times over (row pass at n = 100^3, k = 20: 26 -> 22 us).
template <class T>
__host__ __device__ constexpr bool q_blocked(bool natural) { return sizeof(T) == 4 && natural; }
// floats of n rows of kp values in that layout
__host__ __device__ inline int64_t q_blocked_size(int n, int kp) { return ((int64_t)n + 31) / 32 * 32 * kp; }

// cs: Q is streamed once per step and the step's data exceed L2, so its rows are
// loaded evict-first to keep the reused vectors in L2 (see stream_evict_first)
template <class T, int KP, bool BLK>
__device__ __forceinline__ void load_qrow(const T* __restrict__ Q, int i, T (&q)[KP > 0 ? KP : 1],
                                          bool cs = false) {
    if constexpr (KP > 0) {
        if constexpr (sizeof(T) == 4) {
            // every padded width is a multiple of 4
            const float4* a = BLK ? reinterpret_cast<const float4*>(Q + (size_t)(i & ~31) * KP) + (i & 31)
                                  : reinterpret_cast<const float4*>(Q + (size_t)i * KP);
#pragma unroll
            for (int m = 0; m < KP; m += 4, a += BLK ? 32 : 1) {
                float4 v = cs ? __ldcs(a) : __ldg(a);
                q[m] = v.x;
                q[m + 1] = v.y;
                q[m + 2] = v.z;
                q[m + 3] = v.w;
            }
        } else {
            const T* row = Q + (size_t)i * KP;
#pragma unroll
            for (int m = 0; m < KP; m += 2) {
                double2 v = *reinterpret_cast<const double2*>(row + m);
                q[m] = v.x;
                q[m + 1] = v.y;
            }
        }
    }
}

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Error-free FP32 pair ("double-float") addition: TwoSum of the leading parts, the
// trailing parts added to the error, renormalised.  About 44 significant bits, so
// the FP32 solve's cross-block sums stay accurate without the (slow) FP64 pipe.
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    float s = a.x + b.x;
    float bb = s - a.x;
    float e = (a.x - (s - bb)) + (b.x - bb);
    e += a.y + b.y;
    float hi = s + e;
    float lo = e - (hi - s);
    return make_float2(hi, lo);
}

// Row i of J~ y over skew half-diagonals, G at a time, the 4 G loads of a group ahead of its products
// (Ud: U_0 at the row, yi: y at the row).  The order in which ptxas issues the loads of the
// plain loop changes with everything around it; where that costs, the kernels take this one.
// k_mrs, FP32, G = 12 against the plain loop, solves launch by launch at 115^3: k = 8 2205 -> 2127 us,
// 12 2273 -> 2141, 20 2384 -> 2308, 32 2514 -> 2360, BF16 Q_k 20 2344 -> 2070; at 150^3 k = 20 5131 -> 4928,
// BF16 5126 -> 4281; at 100^3 equal (k = 20 1621 / 1628, BF16 1602 -> 1530).  G = 6 and 8 lose in places.
template <class T, int G>
__device__ __forceinline__ T dia_row(const T* __restrict__ Ud, long long ustride, const T* yi, const int* off,
                                     int ndiag) {
    T acc = (T)0;
    for (int d0 = 0; d0 < ndiag; d0 += G) {
        T ua[G], ub[G], ya[G], yb[G];
#pragma unroll
        for (int u = 0; u < G; ++u) {
            const bool in = d0 + u < ndiag;
            const int m = in ? off[d0 + u] : 0;
            const T* Um = Ud + (in ? d0 + u : 0) * ustride;
            ua[u] = in ? __ldg(Um) : (T)0;
            ub[u] = in ? __ldg(Um - m) : (T)0;
            ya[u] = yi[m];
            yb[u] = yi[-m];
        }
#pragma unroll
        for (int u = 0; u < G; ++u) acc += ua[u] * ya[u] - ub[u] * yb[u];
    }
    return acc;
}

// sum of N values by a balanced tree in a fixed order (log2 N dependent additions)
template <class P, int N, class Add>
__device__ __forceinline__ P pair_tree(P (&a)[N], Add add) {
    static_assert((N & (N - 1)) == 0, "a power of two");
#pragma unroll
    for (int h = N / 2; h > 0; h >>= 1)
#pragma unroll
        for (int i = 0; i < h; ++i) a[i] = add(a[i], a[i + h]);
    return a[0];
}

// Scalar state of the recurrence, kept in shared memory and advanced by one
// thread per block in the precision of the vectors (the FP32 solve keeps its
// whole synchronisation chain off the narrow FP64 pipe of this part; every block
// computes the same values from the same reduced sums, so all blocks agree bit
// for bit).
template <class S>
struct MrsScalars {
    S r0, rr0, nu, coef_old, theta_t, c_prev, s_prev, delta_prev, G;
    S nu_p, delta_pp, rtheta_p, xcoef_p;   // rtheta_p = 1 / theta of the previous step
    // final-pass coefficients when the iteration stops
    S fin_nu, fin_delta, fin_rtheta, fin_xcoef;
    S ratio;
    int its, stop;
};

// block b owns slices [blk[b], blk[b+1]), balanced by stored entries (SELL) or
// uniform (diagonal storage: every row carries the same work)
static __global__ void k_partition(const int* sptr, int nslices, int nblk, int* blk) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nblk) return;
    if (b == nblk) {
        blk[b] = nslices;
        return;
    }
    if (!sptr) {
        blk[b] = (int)((long long)nslices * b / nblk);
        return;
    }
    long long total = sptr[nslices];
    // slices also carry fixed per-row work (Q row, vectors): weight = stored + 32*8
    long long wtot = total + (long long)nslices * 256;
    long long target = wtot * b / nblk;
    int lo = 0, hi = nslices;
    while (lo < hi) {
        int mid = lo + ((hi - lo) >> 1);   // no overflow for offsets near 2^31
        long long w = (long long)sptr[mid] + (long long)mid * 256;
        if (w < target) lo = mid + 1;
        else hi = mid;
    }
    blk[b] = lo;
}

// row-stream storage: block b owns rows [blk[b], blk[b+1]), balanced by stored entries plus
// rowcost a row
static __global__ void k_partition_rows(const int* rp, int n, int rowcost, int nblk, int* blk) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nblk) return;
    if (b == nblk) {
        blk[b] = n;
        return;
    }
    const long long total = (long long)rp[n] + (long long)n * rowcost;
    const long long target = total * b / nblk;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if ((long long)rp[mid] + (long long)mid * rowcost < target) lo = mid + 1;
        else hi = mid;
    }
    blk[b] = lo;
}

}  // namespace asss
