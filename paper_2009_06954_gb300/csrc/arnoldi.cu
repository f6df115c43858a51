// One Arnoldi step of the outer flexible GMRES (§4.1 outer method, reading of
// the FGMRES cycle): given w = A_cal z_j, two classical Gram-Schmidt passes
// against v_0..v_j, the norm of what is left, the Givens update of the Hessenberg
// column and of the residual vector g, and v_{j+1} = w / ||w||, all in one
// cooperative launch with two grid barriers (the passes over V are the only HBM
// traffic; the dot products of a pass are reduced deterministically, every block
// adding the block partials in the same order).  The norm after the second pass
// comes from the one before it: with w1 = w - V h1 and h2 = V^T w1,
// ||w1 - V h2||^2 = ||w1||^2 - ||h2||^2 up to the (re-orthogonalised) departure of V
// from orthonormality, so the second correction and the new basis vector share one
// sweep.
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace asss {

constexpr int AO_WIDE = 512;    // threads of the sweeping kernel
constexpr int AO_TIGHT = 256;   // threads of the register-resident kernel
constexpr int AO_REGV = 6;      // most vectors of the register-resident kernel
constexpr int AO_REGR = 8;      // most rows a thread of it holds

struct AoParams {
    const double* V;  // n x (m+1), column-major (ld n); v_0..v_j are read, v_{j+1} written
    double* w;
    int n, nv;        // nv = j + 1
    int j, m;
    double* H;        // (m+1) x m column-major Hessenberg, already rotated
    double* cs;
    double* sn;
    double* g;
    double* hv;       // first-pass coefficients (nv)
    double* hv2;      // second-pass coefficients (nv)
    double* hn2;      // ||w||^2 after both passes
    double* inv_hn;   // 1 / ||w|| (0 when w = 0)
    double* part;     // 2 x [AO_MAXV][nblk] block partials (consecutive passes alternate halves)
    double thr;       // the cycle stops when |g[j+1]| <= thr
    double sign;      // v_{j+1} = sign * w / ||w||
    int* stop;
    GridBarrier gb;
    unsigned phase0;  // barriers completed on gb.count before this launch
    long long budget;
};

// A warp's FP64 instruction holds its SM quarter's pipe for 64 cycles on this part, so what
// one warp does alone (norms, the Givens update) is written for few dependent operations:
// a square root and its reciprocal come from one rsqrt.
__device__ __forceinline__ void ao_root(double a, double* root, double* inv) {
    const double r = a > 0.0 ? rsqrt(a) : 0.0;
    *root = a * r;
    *inv = r;
}

// Givens update of column j; s_cs, s_sn: the earlier rotations, gj = g[j]
__device__ void ao_fg_column(const AoParams& p, const double* h1, const double* h2, double hn2, double hn, double inv,
                             const double* s_cs, const double* s_sn, double gj) {
    const int j = p.j, m = p.m;
    double* col = p.H + (size_t)j * (m + 1);
    double cur = h1[0] + h2[0];
    for (int a = 0; a < j; ++a) {
        const double next = h1[a + 1] + h2[a + 1];
        col[a] = s_cs[a] * cur + s_sn[a] * next;
        cur = s_cs[a] * next - s_sn[a] * cur;
    }
    const double big = fmax(fabs(cur), hn);
    double rr, c, s;
    if (big > 1e-140 && big < 1e140) {   // the squares neither underflow nor overflow
        double ir;
        ao_root(cur * cur + hn * hn, &rr, &ir);
        c = cur * ir;
        s = hn * ir;
    } else {
        rr = hypot(cur, hn);
        c = (rr != 0.0) ? cur / rr : 1.0;
        s = (rr != 0.0) ? hn / rr : 0.0;
    }
    const double gn = -s * gj;
    p.cs[j] = c;
    p.sn[j] = s;
    col[j] = rr;
    col[j + 1] = 0.0;
    p.g[j + 1] = gn;
    p.g[j] = c * gj;
    *p.hn2 = hn2;
    *p.inv_hn = inv;
    *p.stop = (hn2 == 0.0 || fabs(gn) <= p.thr) ? 1 : 0;
}

// s_out[a] = sum over blocks of part[a][block] for a < cnt, one warp per value (in the same
// order in every block); the caller synchronises
template <int NT>
__device__ __forceinline__ void ao_reduce(const double* part, int cnt, int nblk, double* s_out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int a = warp; a < cnt; a += NT / 32) {
        double t = 0.0;
        for (int b0 = 0; b0 < nblk; b0 += 160) {   // up to five loads in flight
            double ld[5];
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const int b = b0 + lane + 32 * u;
                ld[u] = b < nblk ? __ldcg(&part[(size_t)a * nblk + b]) : 0.0;
            }
            t += (ld[0] + ld[1]) + (ld[2] + ld[3]) + ld[4];
        }
        t = warp_sum(t);
        if (lane == 0) s_out[a] = t;
    }
}

// what closes a step, once s_h2[0..nv) and s_h2[nv] = ||w1||^2 stand in shared memory: warp 0
// forms the norm, rows run row(inv) between, block 0 writes the Hessenberg column
// (hn2 = ||w1||^2 - ||h2||^2)
template <class Rows, class Out>
__device__ __forceinline__ void ao_close(const AoParams& p, const double* s_h1, const double* s_h2, double* s_fin,
                                         const double* s_cs, const double* s_sn, double gj, Rows rows, Out out) {
    if (threadIdx.x < 32) {
        double h2n = 0.0;
        for (int a = 0; a < p.nv; ++a) h2n += s_h2[a] * s_h2[a];
        const double hn2 = fmax(s_h2[p.nv] - h2n, 0.0);
        double hn, inv;
        ao_root(hn2, &hn, &inv);
        if (threadIdx.x == 0) {
            s_fin[0] = hn2;
            s_fin[1] = hn;
            s_fin[2] = inv;
        }
    }
    rows();
    __syncthreads();
    out(p.sign * s_fin[2]);
    if (blockIdx.x == 0) {
        for (int a = threadIdx.x; a < p.nv; a += blockDim.x) {
            p.hv[a] = s_h1[a];
            p.hv2[a] = s_h2[a];
        }
        if (threadIdx.x == blockDim.x - 1)
            ao_fg_column(p, s_h1, s_h2, s_fin[0], s_fin[1], s_fin[2], s_cs, s_sn, gj);
    }
}

// Few vectors and few rows per SM: every thread keeps its R rows of w and of the NVC vectors
// in registers through the three passes, which are read once and all at the start (up to
// R (NVC + 1) loads in flight).  8 warps a block: the FP64 pipe needs no more, and each warp
// costs its share of FP64 adds in the block's sums.  Bound: the chain of two grid barriers
// with their sums.  It serves the Lanczos set-up and FGMRES launch by launch (restarts above 60,
// general patterns; the whole-solve kernel has its own step).  Mean over the steps of a
// launch-by-launch solve, against the sweeping kernel this replaced at these sizes: n = 10^3
// 22 -> 12 us, 47^3 29 -> 17 us, 64^3 36 -> 22 us.
template <int NVC, int R>
__global__ void __launch_bounds__(AO_TIGHT, 1) k_arnoldi_tight(AoParams p) {
    __shared__ double s_w[AO_TIGHT / 32][NVC + 1];
    __shared__ double s_h1[NVC + 1], s_h2[NVC + 1], s_fin[3], s_cs[NVC], s_sn[NVC];
    const int warp = threadIdx.x >> 5;
    const int nblk = gridDim.x;
    const long long n = p.n;
    const int r0 = (int)(n * blockIdx.x / nblk), r1 = (int)(n * (blockIdx.x + 1) / nblk);
    const int nact = min(AO_TIGHT / 32, (r1 - r0 + 31) >> 5);   // warps with rows
    double wi[R], vi[NVC][R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r0 + threadIdx.x + r * AO_TIGHT;
        const bool in = i < r1;
        wi[r] = in ? p.w[i] : 0.0;
#pragma unroll
        for (int t = 0; t < NVC; ++t) vi[t][r] = in ? p.V[(size_t)t * n + i] : 0.0;
    }
    double gj = 0.0;
    if (blockIdx.x == 0) {   // the earlier rotations, long before they are needed
        if (threadIdx.x < NVC && (int)threadIdx.x < p.j) {
            s_cs[threadIdx.x] = p.cs[threadIdx.x];
            s_sn[threadIdx.x] = p.sn[threadIdx.x];
        }
        gj = p.g[p.j];
    }
    auto partials = [&](auto& acc, double* part) {
        constexpr int CNT = sizeof(acc) / sizeof(double);
        if (warp < nact) warp_fold_to<CNT>(acc, s_w[warp]);
        __syncthreads();
        if (threadIdx.x < CNT) {
            double s = 0.0;
            for (int q = 0; q < nact; ++q) s += s_w[q][threadIdx.x];
            part[(size_t)threadIdx.x * nblk + blockIdx.x] = s;
        }
    };
    // ---- pass 1: h1 = V^T w ----
    {
        double acc[NVC];
#pragma unroll
        for (int t = 0; t < NVC; ++t) {
            acc[t] = 0.0;
#pragma unroll
            for (int r = 0; r < R; ++r) acc[t] += vi[t][r] * wi[r];
        }
        partials(acc, p.part);
    }
    if (!grid_sync_phase(p.gb, nblk, p.phase0 + 0, p.budget)) return;
    ao_reduce<AO_TIGHT>(p.part, NVC, nblk, s_h1);
    __syncthreads();
    // ---- pass 2: w1 = w - V h1, h2 = V^T w1, ||w1||^2 ----
    double* part2 = p.part + (size_t)AO_MAXV * nblk;
    {
        double acc[NVC + 1];
#pragma unroll
        for (int t = 0; t <= NVC; ++t) acc[t] = 0.0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double s = 0.0;
#pragma unroll
            for (int t = 0; t < NVC; ++t) s += vi[t][r] * s_h1[t];
            wi[r] -= s;
#pragma unroll
            for (int t = 0; t < NVC; ++t) acc[t] += vi[t][r] * wi[r];
            acc[NVC] += wi[r] * wi[r];
        }
        partials(acc, part2);
    }
    if (!grid_sync_phase(p.gb, nblk, p.phase0 + 1, p.budget)) return;
    ao_reduce<AO_TIGHT>(part2, NVC + 1, nblk, s_h2);
    __syncthreads();
    // ---- pass 3: w2 = w1 - V h2, v_{j+1} = w2 / ||w2|| ----
    ao_close(p, s_h1, s_h2, s_fin, s_cs, s_sn, gj,
             [&]() {
#pragma unroll
                 for (int r = 0; r < R; ++r) {
                     double s = 0.0;
#pragma unroll
                     for (int t = 0; t < NVC; ++t) s += vi[t][r] * s_h2[t];
                     wi[r] -= s;
                 }
             },
             [&](double inv) {
                 double* vn = const_cast<double*>(p.V) + (size_t)NVC * n;
#pragma unroll
                 for (int r = 0; r < R; ++r) {
                     const int i = r0 + threadIdx.x + r * AO_TIGHT;
                     if (i < r1) {
                         p.w[i] = wi[r];
                         vn[i] = wi[r] * inv;
                     }
                 }
             });
}

// Any number of vectors and rows: three sweeps over the block's rows of V and w.  Up to
// AO_REGV vectors a row's dot products run together, U rows at a time, so that U (nv + 1) loads
// are in flight; above that the dot products are spread over the warps (a warp takes a vector,
// or a share of its rows) and need no sums across warps in registers: 41 -> 19 us a step at
// n = 20011 over 15 steps; 56 -> 47 us at 100^3 launch by launch, where FP64 FMAs and bytes need about 20.
__global__ void __launch_bounds__(AO_WIDE, 1) k_arnoldi_orth(AoParams p) {
    constexpr int NW = AO_WIDE / 32;
    __shared__ double s_w[NW][AO_REGV + 1];
    __shared__ double s_h1[AO_MAXV], s_h2[AO_MAXV + 1], s_fin[3], s_cs[AO_MAXV], s_sn[AO_MAXV];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = gridDim.x;
    const long long n = p.n;
    const int r0 = (int)(n * blockIdx.x / nblk), r1 = (int)(n * (blockIdx.x + 1) / nblk);
    const int nact = min(NW, (r1 - r0 + 31) >> 5);
    const int nv = p.nv;
    const double* __restrict__ V = p.V;  // v_0..v_j (read) and v_{j+1} (written) do not overlap w
    double* __restrict__ w = p.w;
    double gj = 0.0;
    if (blockIdx.x == 0) {
        for (int a = threadIdx.x; a < p.j; a += AO_WIDE) {
            s_cs[a] = p.cs[a];
            s_sn[a] = p.sn[a];
        }
        gj = p.g[p.j];
    }
    // block sums of the accumulators; value t to slot t of part, or all to slot `slot`
    auto partials = [&](auto& acc, double* part, int slot) {
        constexpr int CNT = sizeof(acc) / sizeof(double);
        if (warp < nact) warp_fold_to<CNT>(acc, s_w[warp]);
        __syncthreads();
        if (threadIdx.x < CNT) {
            double s = 0.0;
            for (int q = 0; q < nact; ++q) s += s_w[q][threadIdx.x];
            part[(size_t)(slot + threadIdx.x) * nblk + blockIdx.x] = s;
        }
        __syncthreads();
    };
    // f(count as a constant) for the vector counts that are held in registers
    auto by_count = [&](auto f) {
        switch (nv) {
            case 1: f(std::integral_constant<int, 1>{}); break;
            case 2: f(std::integral_constant<int, 2>{}); break;
            case 3: f(std::integral_constant<int, 3>{}); break;
            case 4: f(std::integral_constant<int, 4>{}); break;
            case 5: f(std::integral_constant<int, 5>{}); break;
            default: f(std::integral_constant<int, 6>{}); break;
        }
    };
    // rows in groups of U: load(i, u) for each, then use(i, u)
    auto sweep = [&](auto uc, auto load, auto use) {
        constexpr int U = decltype(uc)::value;
        int i = r0 + threadIdx.x;
        for (; i + (U - 1) * AO_WIDE < r1; i += U * AO_WIDE) {
#pragma unroll
            for (int u = 0; u < U; ++u) load(i + u * AO_WIDE, u);
#pragma unroll
            for (int u = 0; u < U; ++u) use(i + u * AO_WIDE, u);
        }
        for (; i < r1; i += AO_WIDE) {
            load(i, 0);
            use(i, 0);
        }
    };
    // dots of many vectors: wpv warps share a vector (16 / nv of them, at least one); their
    // shares of the rows are summed by one thread
    auto dots_by_warp = [&](double* part) {
        const int wpv = NW / nv > 0 ? NW / nv : 1;
        const int groups = NW / wpv;
        const int grp = warp / wpv, sub = warp % wpv;
        for (int a0 = 0; a0 < nv; a0 += groups) {
            const int a = a0 + grp;
            double t = 0.0;
            if (grp < groups && a < nv) {
                const double* va = V + (size_t)a * n;
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
                int i = r0 + sub * 32 + lane;
                const int st = wpv * 32;
                for (; i + 3 * st < r1; i += 4 * st)
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[u] += va[i + u * st] * w[i + u * st];
                for (; i < r1; i += st) acc[0] += va[i] * w[i];
                t = warp_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
            }
            if (wpv == 1) {
                if (lane == 0 && a < nv) part[(size_t)a * nblk + blockIdx.x] = t;
            } else {
                __syncthreads();
                if (lane == 0) s_w[warp][0] = t;
                __syncthreads();
                if (lane == 0 && sub == 0 && grp < groups && a < nv) {
                    double s = 0.0;
                    for (int q = 0; q < wpv; ++q) s += s_w[warp + q][0];
                    part[(size_t)a * nblk + blockIdx.x] = s;
                }
            }
        }
    };
    // w_i -= sum_a V_ai h_a for one row, the loads of eight vectors in flight
    auto project = [&](int i, const double* h) {
        double s = 0.0;
        for (int a = 0; a < nv; a += 8) {
            double ld[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) ld[u] = a + u < nv ? V[(size_t)(a + u) * n + i] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += ld[u] * h[a + u < nv ? a + u : 0];
        }
        return w[i] - s;
    };
    const bool few = nv <= AO_REGV;

    // ---- pass 1: h1 = V^T w ----
    if (few) {
        by_count([&](auto nvc) {
            constexpr int NVC = decltype(nvc)::value, U = NVC <= 3 ? 4 : 2;
            double acc[NVC], vi[U][NVC], wi[U];
#pragma unroll
            for (int t = 0; t < NVC; ++t) acc[t] = 0.0;
            sweep(std::integral_constant<int, U>{},
                  [&](int i, int u) {
                      wi[u] = w[i];
#pragma unroll
                      for (int t = 0; t < NVC; ++t) vi[u][t] = V[(size_t)t * n + i];
                  },
                  [&](int, int u) {
#pragma unroll
                      for (int t = 0; t < NVC; ++t) acc[t] += vi[u][t] * wi[u];
                  });
            partials(acc, p.part, 0);
        });
    } else {
        dots_by_warp(p.part);
    }
    if (!grid_sync_phase(p.gb, nblk, p.phase0 + 0, p.budget)) return;
    ao_reduce<AO_WIDE>(p.part, nv, nblk, s_h1);
    __syncthreads();

    // ---- pass 2: w1 = w - V h1, then h2 = V^T w1 and ||w1||^2 (slot nv) ----
    double* part2 = p.part + (size_t)AO_MAXV * nblk;   // a block may still be adding the first half
    if (few) {
        by_count([&](auto nvc) {
            constexpr int NVC = decltype(nvc)::value, U = NVC <= 3 ? 4 : 2;
            double acc[NVC + 1], vi[U][NVC], wi[U];
#pragma unroll
            for (int t = 0; t <= NVC; ++t) acc[t] = 0.0;
            sweep(std::integral_constant<int, U>{},
                  [&](int i, int u) {
                      wi[u] = w[i];
#pragma unroll
                      for (int t = 0; t < NVC; ++t) vi[u][t] = V[(size_t)t * n + i];
                  },
                  [&](int i, int u) {
                      double s = 0.0;
#pragma unroll
                      for (int t = 0; t < NVC; ++t) s += vi[u][t] * s_h1[t];
                      const double wn = wi[u] - s;
                      w[i] = wn;
#pragma unroll
                      for (int t = 0; t < NVC; ++t) acc[t] += vi[u][t] * wn;
                      acc[NVC] += wn * wn;
                  });
            partials(acc, part2, 0);
        });
    } else {
        double accn[1] = {0.0};
        for (int i = r0 + threadIdx.x; i < r1; i += AO_WIDE) {
            const double wn = project(i, s_h1);
            w[i] = wn;
            accn[0] += wn * wn;
        }
        partials(accn, part2, nv);   // (its barriers also publish w1 to the block)
        dots_by_warp(part2);
    }
    if (!grid_sync_phase(p.gb, nblk, p.phase0 + 1, p.budget)) return;
    ao_reduce<AO_WIDE>(part2, nv + 1, nblk, s_h2);
    __syncthreads();

    // ---- pass 3: w2 = w1 - V h2 and v_{j+1} = w2 / ||w2|| in one sweep ----
    double* vn = const_cast<double*>(V) + (size_t)nv * n;
    ao_close(p, s_h1, s_h2, s_fin, s_cs, s_sn, gj, [] {},
             [&](double inv) {
                 if (few) {
                     by_count([&](auto nvc) {
                         constexpr int NVC = decltype(nvc)::value, U = NVC <= 3 ? 4 : 2;
                         double vi[U][NVC], wi[U];
                         sweep(std::integral_constant<int, U>{},
                               [&](int i, int u) {
                                   wi[u] = w[i];
#pragma unroll
                                   for (int t = 0; t < NVC; ++t) vi[u][t] = V[(size_t)t * n + i];
                               },
                               [&](int i, int u) {
                                   double s = 0.0;
#pragma unroll
                                   for (int t = 0; t < NVC; ++t) s += vi[u][t] * s_h2[t];
                                   const double wn = wi[u] - s;
                                   w[i] = wn;
                                   vn[i] = wn * inv;
                               });
                     });
                 } else {
                     for (int i = r0 + threadIdx.x; i < r1; i += AO_WIDE) {
                         const double wn = project(i, s_h2);
                         w[i] = wn;
                         vn[i] = wn * inv;
                     }
                 }
             });
}

template <int NVC>
static const void* ao_tight(int rows) {
    return rows <= 1   ? (const void*)k_arnoldi_tight<NVC, 1>
           : rows <= 2 ? (const void*)k_arnoldi_tight<NVC, 2>
           : rows <= 4 ? (const void*)k_arnoldi_tight<NVC, 4>
                       : (const void*)k_arnoldi_tight<NVC, 8>;
}

asss_status arnoldi_orth(const Ctx& c, ArnoldiWork& aw, const double* V, double* w, int n, int j, int m, double* H,
                         double* cs, double* sn, double* g, double* hv, double* hv2, double* hn2, double* inv_hn,
                         double thr, int* stop, double sign) {
    if (j + 1 > AO_MAXV - 1) {   // one partial slot is kept for the norm
        set_error("Arnoldi step %d exceeds the fused kernel's %d vectors", j, AO_MAXV - 1);
        return ASSS_ERR_UNSUPPORTED;
    }
    if (aw.n != n || !aw.part.p) {
        int occ = 0;
        ASSS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_arnoldi_orth, AO_WIDE, 0));
        if (occ < 1) {
            set_error("Arnoldi kernel cannot be resident");
            return ASSS_ERR_CUDA;
        }
        if (occ > 1) occ = 1;
        int nblk = c.sms * occ;
        int need = cdiv(n, 64);
        if (need < 1) need = 1;
        if (nblk > need) nblk = need;
        ASSS_TRY(aw.part.alloc((int64_t)2 * AO_MAXV * nblk));
        if (!aw.bar.p) ASSS_TRY(aw.bar.alloc(2));
        if (!aw.err.p) ASSS_TRY(aw.err.alloc(1));
        ASSS_CUDA(cudaMemsetAsync(aw.bar.p, 0, 2 * sizeof(unsigned), c.stream));
        ASSS_CUDA(cudaMemsetAsync(aw.err.p, 0, sizeof(int), c.stream));
        aw.nblk = nblk;
        aw.n = n;
        aw.phase = 0;
    }
    AoParams p;
    p.V = V;
    p.w = w;
    p.n = n;
    p.nv = j + 1;
    p.j = j;
    p.m = m;
    p.H = H;
    p.cs = cs;
    p.sn = sn;
    p.g = g;
    p.hv = hv;
    p.hv2 = hv2;
    p.hn2 = hn2;
    p.inv_hn = inv_hn;
    p.part = aw.part.p;
    p.thr = thr;
    p.sign = sign;
    p.stop = stop;
    p.gb.count = aw.bar.p;
    p.gb.err = aw.err.p;
    p.phase0 = aw.phase;
    p.budget = c.wait_cycles;
    void* args[] = {&p};
    // rows a thread of the register-resident kernel would hold, and its instantiation
    const int rows = cdiv(cdiv(n, aw.nblk), AO_TIGHT);
    const void* fn = (const void*)k_arnoldi_orth;
    int nt = AO_WIDE;
    if (p.nv <= AO_REGV && rows <= AO_REGR) {
        nt = AO_TIGHT;
        switch (p.nv) {
            case 1: fn = ao_tight<1>(rows); break;
            case 2: fn = ao_tight<2>(rows); break;
            case 3: fn = ao_tight<3>(rows); break;
            case 4: fn = ao_tight<4>(rows); break;
            case 5: fn = ao_tight<5>(rows); break;
            default: fn = ao_tight<6>(rows); break;
        }
    }
    ASSS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(aw.nblk), dim3(nt), args, 0, c.stream));
    count_launch();
    aw.phase += 2;
    return ASSS_OK;
}

}  // namespace asss
