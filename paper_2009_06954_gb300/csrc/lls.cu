// The least-squares problem for the shifted skew-symmetrizer S (paper §2,
// Eqs. eq1, eq2, regularized; App. A), solved on the device without forming B.
//
// Unknowns: the entries of S on its pattern (CSR order).  Constraint rows: one
// per upper entry (i < j) of the symmetric pattern P = pat(Abar S) + pat(Abar S)^T,
// stating (Abar S)_ij + (Abar S)_ji = 0, and one per diagonal entry,
// sqrt(gamma) (Abar S)_ii = sqrt(gamma).  With C = Abar S evaluated on P:
//   (B s)_ij = C_ij + C_ji  (i < j),    (B s)_ii = sqrt(gamma) C_ii
//   (B^T t)_lj = sum_i abar_il G_ij  with G symmetric on P, G_ij = t_{min,max}
//   (off-diagonal) and G_ii = sqrt(gamma) t_ii.
// Each output is one sorted-list intersection ("merge dot"), computed by one
// thread, so results do not depend on scheduling.
//
// The normal equations B^T B s = B^T v are solved by preconditioned conjugate
// gradients.  The preconditioner is block-Jacobi on the pairs {s_lj, s_jl}: when
// Abar is close to I a skew perturbation of S barely changes the objective, so
// the two entries of a pair are strongly coupled; the 2x2 Gram block of a pair is
//   [ sum_i abar_il^2 w_ij     abar_ll abar_jj ]
//   [ abar_ll abar_jj          sum_i abar_ij^2 w_il ]     (w = gamma on i = column)
// and is inverted in closed form.
#include "common.cuh"
#include "internal.h"

namespace asss {

__device__ __forceinline__ double merge_dot_s(const int* __restrict__ ac, const double* __restrict__ av, int alen,
                                              const int* __restrict__ bc, const int* __restrict__ bu, int blen,
                                              const double* __restrict__ s) {
    int x = 0, y = 0;
    double acc = 0.0;
    while (x < alen && y < blen) {
        int ca = ac[x], cb = bc[y];
        if (ca == cb) {
            acc += av[x] * s[bu[y]];
            ++x;
            ++y;
        } else if (ca < cb) {
            ++x;
        } else {
            ++y;
        }
    }
    return acc;
}

__global__ void k_row_of_entry(const int* rp, int n, int* row) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int e = rp[i]; e < rp[i + 1]; ++e) row[e] = i;
}

// q = B s on the constraint entries of P (upper + diagonal); lower entries get 0
__global__ void k_lls_B(int nP, const int* __restrict__ prow, const int* __restrict__ pci,
                        const int* __restrict__ arp, const int* __restrict__ aci, const double* __restrict__ av,
                        const int* __restrict__ strp, const int* __restrict__ stci, const int* __restrict__ stsrc,
                        const double* __restrict__ s, double sg, double* q) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nP) return;
    int i = prow[k], j = pci[k];
    if (j < i) {
        q[k] = 0.0;
        return;
    }
    double cij = merge_dot_s(aci + arp[i], av + arp[i], arp[i + 1] - arp[i], stci + strp[j], stsrc + strp[j],
                             strp[j + 1] - strp[j], s);
    if (j == i) {
        q[k] = sg * cij;
        return;
    }
    double cji = merge_dot_s(aci + arp[j], av + arp[j], arp[j + 1] - arp[j], stci + strp[i], stsrc + strp[i],
                             strp[i + 1] - strp[i], s);
    q[k] = cij + cji;
}

// C = Abar S on every entry of P
__global__ void k_lls_C(int nP, const int* __restrict__ prow, const int* __restrict__ pci,
                        const int* __restrict__ arp, const int* __restrict__ aci, const double* __restrict__ av,
                        const int* __restrict__ strp, const int* __restrict__ stci, const int* __restrict__ stsrc,
                        const double* __restrict__ s, double* C) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nP) return;
    int i = prow[k], j = pci[k];
    C[k] = merge_dot_s(aci + arp[i], av + arp[i], arp[i + 1] - arp[i], stci + strp[j], stsrc + strp[j],
                       strp[j + 1] - strp[j], s);
}

// g = B^T t on the unknowns
__global__ void k_lls_BT(int nS, const int* __restrict__ srow, const int* __restrict__ sci,
                         const int* __restrict__ atrp, const int* __restrict__ atci, const double* __restrict__ atv,
                         const int* __restrict__ prp, const int* __restrict__ pci, const int* __restrict__ mirror,
                         const double* __restrict__ t, double sg, double* g) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nS) return;
    int l = srow[u], j = sci[u];
    int x = atrp[l], xe = atrp[l + 1];
    int y = prp[j], ye = prp[j + 1];
    double acc = 0.0;
    while (x < xe && y < ye) {
        int ia = atci[x], ib = pci[y];
        if (ia == ib) {
            double G;
            if (ia > j) G = t[y];
            else if (ia < j) G = (mirror[y] >= 0) ? t[mirror[y]] : 0.0;
            else G = sg * t[y];
            acc += atv[x] * G;
            ++x;
            ++y;
        } else if (ia < ib) {
            ++x;
        } else {
            ++y;
        }
    }
    g[u] = acc;
}

// ---------------------------------------------------------------------------
// B and B^T stored explicitly (when they fit a memory budget) in SELL slices of 32 rows: the
// entries each merge above would visit, in the same order, so an iteration streams two
// sparse matrices instead of redoing the intersections.
//   B: one row per constraint (the upper and diagonal entries of P; the lower ones are left
//   out), in slots sorted by length within windows; the weight sqrt(gamma) of the diagonal
//   constraints is in the values.
//   B^T: one row per unknown, the two unknowns of a preconditioner pair in neighbouring slots
//   (2t, 2t + 1), so that the lane next door holds the partner's residual.
// All vectors of the iteration stand in these slot orders.
// ---------------------------------------------------------------------------
// entries of the intersection: count (oc == nullptr) or fill with stride 32, columns through map
__device__ __forceinline__ int merge_list(const int* __restrict__ ac, const double* __restrict__ av, int alen,
                                          const int* __restrict__ bc, const int* __restrict__ bu, int blen,
                                          const int* __restrict__ map, double f, int* oc, double* ov) {
    int x = 0, y = 0, k = 0;
    while (x < alen && y < blen) {
        int ca = ac[x], cb = bc[y];
        if (ca == cb) {
            if (oc) {
                oc[k * 32] = map[bu[y]];
                ov[k * 32] = f * av[x];
            }
            ++k;
            ++x;
            ++y;
        } else if (ca < cb) {
            ++x;
        } else {
            ++y;
        }
    }
    return k;
}

// entries of each row of B (0 for the lower entries of P) and the constraint flags
__global__ void k_bx_count(int nP, const int* __restrict__ prow, const int* __restrict__ pci,
                           const int* __restrict__ arp, const int* __restrict__ aci, const double* __restrict__ av,
                           const int* __restrict__ strp, const int* __restrict__ stci, const int* __restrict__ stsrc,
                           int* bcnt, int* flag) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nP) return;
    const int i = prow[k], j = pci[k];
    int c = 0;
    if (j >= i) {
        c = merge_list(aci + arp[i], av + arp[i], arp[i + 1] - arp[i], stci + strp[j], stsrc + strp[j],
                       strp[j + 1] - strp[j], nullptr, 1.0, nullptr, nullptr);
        if (j != i)
            c += merge_list(aci + arp[j], av + arp[j], arp[j + 1] - arp[j], stci + strp[i], stsrc + strp[i],
                            strp[i + 1] - strp[i], nullptr, 1.0, nullptr, nullptr);
    }
    bcnt[k] = c;
    flag[k] = j >= i ? 1 : 0;
}
// constraint c is entry klist[c] of P, with len[c] entries
__global__ void k_bx_list(int nP, const int* flag, const int* cidx, const int* bcnt, int* klist, int* len) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nP || !flag[k]) return;
    klist[cidx[k]] = k;
    len[cidx[k]] = bcnt[k];
}
// a slot's row of B and its start value of rho (the right-hand side v)
__global__ void k_bx_fill(int nslots, int nC, const int* __restrict__ rowmap, const int* __restrict__ klist,
                          const int* __restrict__ prow, const int* __restrict__ pci, const int* __restrict__ arp,
                          const int* __restrict__ aci, const double* __restrict__ av, const int* __restrict__ strp,
                          const int* __restrict__ stci, const int* __restrict__ stsrc, const int* __restrict__ upos,
                          double sg, const int* __restrict__ sptr, int* col, double* val, double* rho) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= nslots) return;
    const int c = rowmap ? rowmap[slot] : slot;
    const int b = sptr[slot >> 5], width = (sptr[(slot >> 5) + 1] - b) >> 5;
    int* oc = col + b + (slot & 31);
    double* ov = val + b + (slot & 31);
    int m = 0;
    double r = 0.0;
    if (c < nC) {
        const int k = klist[c], i = prow[k], j = pci[k];
        m = merge_list(aci + arp[i], av + arp[i], arp[i + 1] - arp[i], stci + strp[j], stsrc + strp[j],
                       strp[j + 1] - strp[j], upos, j == i ? sg : 1.0, oc, ov);
        if (j != i)
            m += merge_list(aci + arp[j], av + arp[j], arp[j + 1] - arp[j], stci + strp[i], stsrc + strp[i],
                            strp[i + 1] - strp[i], upos, 1.0, oc + m * 32, ov + m * 32);
        r = j == i ? sg : 0.0;
    }
    for (; m < width; ++m) {
        oc[m * 32] = 0;
        ov[m * 32] = 0.0;
    }
    rho[slot] = r;
}

// pairs first (slots 2t, 2t + 1), then the unknowns without a partner
__global__ void k_pair_flags(int nS, const int* partner, int* lead, int* single) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nS) return;
    const int p = partner[u];
    lead[u] = p > u ? 1 : 0;
    single[u] = p < 0 ? 1 : 0;
}
// (pmap, smap: places of the pairs and of the single unknowns, null for their own order)
__global__ void k_pair_slots(int nS, const int* partner, const int* lpos, const int* spos, const int* pmap,
                             const int* smap, int npairs, int* upos, int* uslot) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nS) return;
    const int p = partner[u];
    const int t = p < 0 ? spos[u] : lpos[p > u ? u : p];   // number of the single unknown or of the pair
    const int slot = p < 0 ? 2 * npairs + (smap ? smap[t] : t) : 2 * (pmap ? pmap[t] : t) + (p > u ? 0 : 1);
    upos[u] = slot;
    uslot[slot] = u;
}
// lengths by pair (the longer of its two rows) and by single unknown, from the lengths by slot
__global__ void k_pair_len(int npairs, int nsingle, const int* tlen, int* plen, int* slen) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < npairs) plen[t] = max(tlen[2 * t], tlen[2 * t + 1]);
    else if (t - npairs < nsingle) slen[t - npairs] = tlen[npairs + t];
}
// walk of row u of B^T (as k_lls_BT): count, or fill with columns in constraint slots
__device__ __forceinline__ int btx_row(int u, const int* __restrict__ srow, const int* __restrict__ sci,
                                       const int* __restrict__ atrp, const int* __restrict__ atci,
                                       const double* __restrict__ atv, const int* __restrict__ prp,
                                       const int* __restrict__ pci, const int* __restrict__ mirror,
                                       const int* __restrict__ cidx, const int* __restrict__ cpos, double sg, int* oc,
                                       double* ov) {
    const int l = srow[u], j = sci[u];
    int x = atrp[l], xe = atrp[l + 1];
    int y = prp[j], ye = prp[j + 1];
    int k = 0;
    while (x < xe && y < ye) {
        const int ia = atci[x], ib = pci[y];
        if (ia == ib) {
            const int pos = ia >= j ? y : mirror[y];   // no mirror: a zero term, left out
            if (pos >= 0) {
                if (oc) {
                    const int c = cidx[pos];
                    oc[k * 32] = cpos ? cpos[c] : c;
                    ov[k * 32] = ia == j ? sg * atv[x] : atv[x];
                }
                ++k;
            }
            ++x;
            ++y;
        } else if (ia < ib) {
            ++x;
        } else {
            ++y;
        }
    }
    return k;
}
__global__ void k_btx_count(int nslots, const int* __restrict__ uslot, const int* srow, const int* sci, const int* atrp,
                            const int* atci, const double* atv, const int* prp, const int* pci, const int* mirror,
                            int* len) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nslots) return;
    const int u = uslot[t];
    len[t] = u < 0 ? 0 : btx_row(u, srow, sci, atrp, atci, atv, prp, pci, mirror, nullptr, nullptr, 1.0, nullptr, nullptr);
}
// a slot's row of B^T, its start value of s and the two coefficients of its preconditioner
// block: z = m1 r + m2 r(partner)
__global__ void k_btx_fill(int nslots, const int* __restrict__ uslot, const int* srow, const int* sci, const int* atrp,
                           const int* atci, const double* atv, const int* prp, const int* pci, const int* mirror,
                           const int* cidx, const int* cpos, double sg, const int* sptr, int* col, double* val,
                           const double* N, const int* partner, const double* cross, const double* s0, double* m1,
                           double* m2, double* s) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nslots) return;
    const int u = uslot[t];
    const int b = sptr[t >> 5], width = (sptr[(t >> 5) + 1] - b) >> 5;
    int* oc = col + b + (t & 31);
    double* ov = val + b + (t & 31);
    int m = 0;
    double c1 = 0.0, c2 = 0.0, sv = 0.0;
    if (u >= 0) {
        m = btx_row(u, srow, sci, atrp, atci, atv, prp, pci, mirror, cidx, cpos, sg, oc, ov);
        const double nu = N[u];
        const int p = partner[u];
        if (nu > 0.0) {
            c1 = 1.0 / nu;
            if (p >= 0) {
                const double np = N[p], c = cross[u], det = nu * np - c * c;
                if (det > 1e-12 * nu * np) {
                    c1 = np / det;
                    c2 = -c / det;
                }
            }
        }
        if (s0) sv = s0[u];
    }
    for (; m < width; ++m) {
        oc[m * 32] = 0;
        ov[m * 32] = 0.0;
    }
    m1[t] = c1;
    m2[t] = c2;
    s[t] = sv;
}
__global__ void k_unslot(int nS, const int* upos, const double* s, double* s_val) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < nS) s_val[u] = s[upos[u]];
}

// ---------------------------------------------------------------------------
// the whole PCG in one cooperative launch.  An iteration was eight launches with rows of three
// to seven entries read one thread a row (85 us at n = 32^3, where its data, all in L2, need
// about 10); here it is four phases between grid barriers, a warp a slice:
//   q = B p, ||q||^2 | rho -= a q, s += a p | r = B^T rho, z = M^-1 r, r.z, ||r||^2 | p = z + b p
// r is not stored (z and the two sums are all that is needed of it).  Bound: the FP64 pipe and
// L2 / HBM reads of the entries (12 bytes each).  An iteration at 10^3: 38 -> 7 us, at 32^3: 85 ->
// 25 us, at 64^3: 437 -> 111 us.  Two blocks an SM at 64 registers and four entries in flight:
// eight spill (set-up at 32^3 19.7 ms against 18.5, at 64^3 105 against 95), one block of 117
// registers is as fast at 32^3 and slower from HBM (140 at 64^3).
// ---------------------------------------------------------------------------
constexpr int PCG_THREADS = 512;
struct PcgParams {
    int nb, nt;                       // slices of B and B^T
    const int *bsp, *bcol, *tsp, *tcol;
    const double *bval, *tval, *m1, *m2;
    double *q, *rho, *p, *z, *s;      // 32 nb, 32 nb, 32 nt, 32 nt, 32 nt
    double* part;                     // 2 x [nblk][2]
    GridBarrier gb;
    long long budget;
    double tol;
    int maxit, has_s0, cs;
    int* its;
    double* rel;
};

__global__ void __launch_bounds__(PCG_THREADS, 2) k_lls_pcg(PcgParams P) {
    constexpr int NW = PCG_THREADS / 32;
    __shared__ double s_w[NW][2];
    __shared__ double s_sum[2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = gridDim.x;
    const int b0 = (int)((long long)P.nb * blockIdx.x / nblk), b1 = (int)((long long)P.nb * (blockIdx.x + 1) / nblk);
    const int t0 = (int)((long long)P.nt * blockIdx.x / nblk), t1 = (int)((long long)P.nt * (blockIdx.x + 1) / nblk);
    unsigned phase = 0;
    int sums = 0;
    // sum of a slice's row over x, four entries in flight
    auto row = [&](const int* sp, const int* col, const double* val, int sl, const double* x) -> double {
        const int b = __ldg(&sp[sl]), width = (__ldg(&sp[sl + 1]) - b) >> 5;
        const int* c = col + b + lane;
        const double* v = val + b + lane;
        double acc = 0.0;
        for (int k = 0; k < width; k += 4) {
            int cc[4];
            double vv[4], g[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = k + u < width;
                cc[u] = in ? (P.cs ? __ldcs(c + (k + u) * 32) : __ldg(c + (k + u) * 32)) : 0;
                vv[u] = in ? (P.cs ? __ldcs(v + (k + u) * 32) : __ldg(v + (k + u) * 32)) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = k + u < width ? x[cc[u]] : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k + u < width) acc += vv[u] * g[u];
        }
        return acc;
    };
    // grid totals of two values a thread into s_sum (a grid barrier); false: gave up
    auto grid_sum = [&](double a, double b) -> bool {
        double v[2] = {a, b};
        warp_fold_to<2>(v, s_w[warp]);
        __syncthreads();
        double* part = P.part + (size_t)(sums++ & 1) * 2 * nblk;
        if (threadIdx.x < 2) {
            double t = 0.0;
            for (int w = 0; w < NW; ++w) t += s_w[w][threadIdx.x];
            part[2 * blockIdx.x + threadIdx.x] = t;
        }
        if (!grid_sync_phase(P.gb, nblk, phase++, P.budget)) return false;
        if (warp < 2) {
            double t = 0.0;
            for (int q = lane; q < nblk; q += 32) t += __ldcg(&part[2 * q + warp]);
            t = warp_sum(t);
            if (lane == 0) s_sum[warp] = t;
        }
        __syncthreads();
        return true;
    };
    auto residual = [&]() -> bool {   // z = M^-1 B^T rho; s_sum = r.z, ||r||^2
        double rz = 0.0, rr = 0.0;
        for (int sl = t0 + warp; sl < t1; sl += NW) {
            const int t = sl * 32 + lane;
            const double r = row(P.tsp, P.tcol, P.tval, sl, P.rho);
            const double ro = __shfl_xor_sync(0xffffffffu, r, 1);
            const double zv = P.m1[t] * r + P.m2[t] * ro;
            P.z[t] = zv;
            rz += r * zv;
            rr += r * r;
        }
        return grid_sum(rz, rr);
    };
    // the tolerance is relative to ||B^T v||, the gradient at s = 0, also from given values s0
    if (!residual()) return;
    const double rr0 = s_sum[1];
    double rz = s_sum[0], rel = rr0 > 0.0 ? 1.0 : 0.0;
    if (P.has_s0 && rr0 > 0.0) {   // rho = v - B s0 (the slots of a warp are its own)
        for (int sl = b0 + warp; sl < b1; sl += NW) P.rho[sl * 32 + lane] -= row(P.bsp, P.bcol, P.bval, sl, P.s);
        if (!grid_sync_phase(P.gb, nblk, phase++, P.budget)) return;
        if (!residual()) return;
        rz = s_sum[0];
        rel = sqrt(s_sum[1] / rr0);
    }
    for (int sl = t0 + warp; sl < t1; sl += NW) P.p[sl * 32 + lane] = P.z[sl * 32 + lane];
    if (!grid_sync_phase(P.gb, nblk, phase++, P.budget)) return;
    int its = 0;
    while (rr0 > 0.0 && rel > P.tol && its < P.maxit) {
        double qq = 0.0;
        for (int sl = b0 + warp; sl < b1; sl += NW) {
            const double v = row(P.bsp, P.bcol, P.bval, sl, P.p);
            P.q[sl * 32 + lane] = v;
            qq += v * v;
        }
        if (!grid_sum(qq, 0.0)) return;
        const double a = s_sum[0] > 0.0 ? rz / s_sum[0] : 0.0;
#pragma unroll 4
        for (int sl = b0 + warp; sl < b1; sl += NW) P.rho[sl * 32 + lane] -= a * P.q[sl * 32 + lane];
#pragma unroll 4
        for (int sl = t0 + warp; sl < t1; sl += NW) P.s[sl * 32 + lane] += a * P.p[sl * 32 + lane];
        if (!grid_sync_phase(P.gb, nblk, phase++, P.budget)) return;
        if (!residual()) return;
        const double b = rz != 0.0 ? s_sum[0] / rz : 0.0;
        rz = s_sum[0];
#pragma unroll 4
        for (int sl = t0 + warp; sl < t1; sl += NW) P.p[sl * 32 + lane] = P.z[sl * 32 + lane] + b * P.p[sl * 32 + lane];
        ++its;
        if (its % 8 == 0 || its == P.maxit) {
            rel = sqrt(s_sum[1] / rr0);
            if (rel <= P.tol) break;
        }
        if (!grid_sync_phase(P.gb, nblk, phase++, P.budget)) return;
    }
    if (!(rr0 > 0.0))   // no gradient at s = 0: S = 0, whatever was given
        for (int sl = t0 + warp; sl < t1; sl += NW) P.s[sl * 32 + lane] = 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *P.its = its;
        *P.rel = rel;
    }
}

__global__ void k_diag_values(const int* rp, const int* ci, const double* v, int n, double* dv) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double d = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e)
        if (ci[e] == i) {
            d = v[e];
            break;
        }
    dv[i] = d;
}

__global__ void k_lls_prec_setup(int nS, const int* srow, const int* sci, const int* srp,
                                 const int* atrp, const int* atci, const double* atv, const double* adiag,
                                 double gamma, double* N, int* partner, double* cross) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nS) return;
    int l = srow[u], j = sci[u];
    double acc = 0.0;
    for (int e = atrp[l]; e < atrp[l + 1]; ++e) {
        double a = atv[e];
        acc += a * a * (atci[e] == j ? gamma : 1.0);
    }
    N[u] = acc;
    int p = -1;
    if (l != j) {
        int lo = srp[j], hi = srp[j + 1] - 1;
        while (lo <= hi) {
            int mid = lo + ((hi - lo) >> 1);   // no overflow for offsets near 2^31
            int c = sci[mid];
            if (c == l) {
                p = mid;
                break;
            }
            if (c < l) lo = mid + 1;
            else hi = mid - 1;
        }
    }
    partner[u] = p;
    cross[u] = (p >= 0) ? adiag[l] * adiag[j] : 0.0;
}

__global__ void k_lls_prec_apply(int nS, const double* N, const int* partner, const double* cross, const double* r,
                                 double* z) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nS) return;
    double nu = N[u];
    if (nu <= 0.0) {
        z[u] = 0.0;
        return;
    }
    int p = partner[u];
    if (p >= 0) {
        double np = N[p], c = cross[u];
        double det = nu * np - c * c;
        if (det > 1e-12 * nu * np) {
            z[u] = (np * r[u] - c * r[p]) / det;
            return;
        }
    }
    z[u] = r[u] / nu;
}

__global__ void k_lls_init_rho(int nP, const int* prow, const int* pci, double sg, double* rho) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nP) return;
    rho[k] = (prow[k] == pci[k]) ? sg : 0.0;
}

__global__ void k_cg_update(double* s, const double* p, int nS, double* rho, const double* q, int nP,
                            const double* rz, const double* qq) {
    double a = (*qq > 0.0) ? (*rz) / (*qq) : 0.0;
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nS) s[t] += a * p[t];
    if (t < nP) rho[t] -= a * q[t];
}

__global__ void k_cg_newp(double* p, const double* z, int nS, const double* rz_new, const double* rz_old) {
    double b = (*rz_old != 0.0) ? (*rz_new) / (*rz_old) : 0.0;
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < nS) p[u] = z[u] + b * p[u];
}

__global__ void k_sum_counts(const int* cnt, int n, unsigned long long* total) {
    unsigned long long a = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) a += (unsigned)cnt[i];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(total, a);
}

// the sum of n counts in 64 bits (integer: the same whatever the order)
static asss_status sum_counts(const int* cnt, int n, int64_t* total, cudaStream_t s) {
    DBuf<unsigned long long> t;
    ASSS_TRY(t.alloc(1));
    ASSS_CUDA(cudaMemsetAsync(t.p, 0, sizeof(unsigned long long), s));
    k_sum_counts<<<256, 256, 0, s>>>(cnt, n, t.p);
    ASSS_CHECK_LAUNCH();
    unsigned long long h = 0;
    ASSS_CUDA(cudaMemcpyAsync(&h, t.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    ASSS_CUDA(cudaStreamSynchronize(s));
    *total = (int64_t)h;
    return ASSS_OK;
}

asss_status lls_product_on_pattern(const Ctx& c, const DCsr& Abar, const DCsr& ST, const int* st_src,
                                   const double* s_val, const DCsr& P, const int* prow, double* Cval) {
    k_lls_C<<<cdiv(P.nnz, 256), 256, 0, c.stream>>>(P.nnz, prow, P.ci.p, Abar.rp.p, Abar.ci.p, Abar.v.p, ST.rp.p,
                                                      ST.ci.p, st_src, s_val, Cval);
    ASSS_CHECK_LAUNCH();
    return ASSS_OK;
}

// slice offsets of rows in the given order; sptr stays empty when the total exceeds 32 bits
__global__ void k_slice_width(const int* len, int ns, int* w) {
    const int sl = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (sl >= ns) return;
    int m = len[sl * 32 + lane];
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) w[sl] = m * 32;
}
static asss_status pair_layout(const int* len, int nslots, DBuf<int>& sptr, int64_t* total, cudaStream_t s) {
    const int ns = nslots / 32;
    DBuf<int> w;
    DBuf<long long> off64;
    ASSS_TRY(w.alloc(ns > 0 ? ns : 1));
    ASSS_TRY(off64.alloc(ns + 1));
    sptr.free();
    k_slice_width<<<cdiv(32LL * ns, 256), 256, 0, s>>>(len, ns, w.p);
    ASSS_CHECK_LAUNCH();
    long long tot = 0;
    ASSS_TRY(exclusive_scan64(w.p, off64.p, ns, &tot, s));
    *total = tot;
    if (tot >= (1LL << 31) - 1) return ASSS_OK;
    ASSS_TRY(sptr.alloc(ns + 1));
    ASSS_TRY(exclusive_scan(w.p, sptr.p, ns, nullptr, s));
    ASSS_CUDA(cudaStreamSynchronize(s));   // w is freed here
    return ASSS_OK;
}

asss_status lls_fit(const Ctx& c, const DCsr& Abar, const DCsr& AbarT, const DCsr& Spat, double gamma, double tol,
                    int maxit, DBuf<double>& s_val, DCsr& P, DBuf<int>& mirror, DBuf<int>& diagpos,
                    DBuf<double>& Cval, LlsResult* res, const double* s0) {
    cudaStream_t s = c.stream;
    int n = Abar.n;
    int nS = Spat.nnz;
    // S^T pattern with the CSR position of every entry of S
    DCsr ST;
    DBuf<int> st_src;
    ASSS_TRY(transpose_csr(Spat, ST, &st_src, s));
    ASSS_TRY(build_pattern(Abar, AbarT, Spat, ST, P, mirror, diagpos, s));
    int nP = P.nnz;
    DBuf<int> prow, srow;
    ASSS_TRY(prow.alloc(nP));
    ASSS_TRY(srow.alloc(nS));
    k_row_of_entry<<<cdiv(n, 256), 256, 0, s>>>(P.rp.p, n, prow.p);
    ASSS_CHECK_LAUNCH();
    k_row_of_entry<<<cdiv(n, 256), 256, 0, s>>>(Spat.rp.p, n, srow.p);
    ASSS_CHECK_LAUNCH();

    // preconditioner
    DBuf<double> adiag, Nn, cross;
    DBuf<int> partner;
    ASSS_TRY(adiag.alloc(n));
    ASSS_TRY(Nn.alloc(nS));
    ASSS_TRY(cross.alloc(nS));
    ASSS_TRY(partner.alloc(nS));
    k_diag_values<<<cdiv(n, 256), 256, 0, s>>>(Abar.rp.p, Abar.ci.p, Abar.v.p, n, adiag.p);
    ASSS_CHECK_LAUNCH();
    k_lls_prec_setup<<<cdiv(nS, 256), 256, 0, s>>>(nS, srow.p, Spat.ci.p, Spat.rp.p, AbarT.rp.p, AbarT.ci.p,
                                                    AbarT.v.p, adiag.p, gamma, Nn.p, partner.p, cross.p);
    ASSS_CHECK_LAUNCH();

    const double sg = sqrt(gamma);
    // B and B^T stored explicitly when they fit min(8 GiB, a quarter of the free device
    // memory) with their slices' padding and the iteration's vectors, and the whole iteration in
    // one launch; otherwise the merge kernels apply them matrix-free (ASSS_LLS_STORE_BYTES: another
    // bound)
    {
        DBuf<int> bcnt, cflag, cidx, uslot, upos, lead, single, lpos, spos, tlen;
        ASSS_TRY(bcnt.alloc(nP > 0 ? nP : 1));
        ASSS_TRY(cflag.alloc(nP > 0 ? nP : 1));
        ASSS_TRY(cidx.alloc(nP + 1));
        k_bx_count<<<cdiv(nP, 256), 256, 0, s>>>(nP, prow.p, P.ci.p, Abar.rp.p, Abar.ci.p, Abar.v.p, ST.rp.p, ST.ci.p,
                                                  st_src.p, bcnt.p, cflag.p);
        ASSS_CHECK_LAUNCH();
        int64_t nC = 0, npairs = 0, nsingle = 0, nb = 0, nt = 0, bt = 0, tt = 0;
        ASSS_TRY(exclusive_scan(cflag.p, cidx.p, nP, &nC, s));
        ASSS_TRY(lead.alloc(nS));
        ASSS_TRY(single.alloc(nS));
        ASSS_TRY(lpos.alloc(nS + 1));
        ASSS_TRY(spos.alloc(nS + 1));
        k_pair_flags<<<cdiv(nS, 256), 256, 0, s>>>(nS, partner.p, lead.p, single.p);
        ASSS_CHECK_LAUNCH();
        ASSS_TRY(exclusive_scan(lead.p, lpos.p, nS, &npairs, s));
        ASSS_TRY(exclusive_scan(single.p, spos.p, nS, &nsingle, s));
        const int nuslots = cdiv(2 * npairs + nsingle, 32) * 32;
        const int nbs = cdiv(nC, 32), nts = nuslots / 32;
        ASSS_TRY(upos.alloc(nS));
        ASSS_TRY(uslot.alloc(nuslots));
        ASSS_TRY(tlen.alloc(nuslots));
        // slots of the unknowns (pmap, smap: see k_pair_slots) and the lengths of their rows of B^T
        auto place = [&](const int* pmap, const int* smap) -> asss_status {
            ASSS_CUDA(cudaMemsetAsync(uslot.p, 0xff, sizeof(int) * (size_t)nuslots, s));
            k_pair_slots<<<cdiv(nS, 256), 256, 0, s>>>(nS, partner.p, lpos.p, spos.p, pmap, smap, (int)npairs, upos.p,
                                                        uslot.p);
            ASSS_CHECK_LAUNCH();
            k_btx_count<<<cdiv(nuslots, 256), 256, 0, s>>>(nuslots, uslot.p, srow.p, Spat.ci.p, AbarT.rp.p, AbarT.ci.p,
                                                            AbarT.v.p, P.rp.p, P.ci.p, mirror.p, tlen.p);
            ASSS_CHECK_LAUNCH();
            return ASSS_OK;
        };
        ASSS_TRY(place(nullptr, nullptr));
        ASSS_TRY(sum_counts(bcnt.p, nP, &nb, s));
        ASSS_TRY(sum_counts(tlen.p, nuslots, &nt, s));
        size_t fr = 0, tot = 0;
        ASSS_CUDA(cudaMemGetInfo(&fr, &tot));
        const char* bound = getenv("ASSS_LLS_STORE_BYTES");
        const double budget = bound ? atof(bound) : fmin(8.0 * 1024 * 1024 * 1024, 0.25 * (double)fr);
        const double vectors = 8.0 * (5.0 * nuslots + 2.0 * 32 * nbs);
        DBuf<int> klist, blen, bmap, bpos, bsp, tsp;
        if (12.0 * (double)(nb + nt) + vectors <= budget) {   // else the padded form is above it too
            ASSS_TRY(klist.alloc(nC));
            ASSS_TRY(blen.alloc(nC));
            k_bx_list<<<cdiv(nP, 256), 256, 0, s>>>(nP, cflag.p, cidx.p, bcnt.p, klist.p, blen.p);
            ASSS_CHECK_LAUNCH();
            ASSS_TRY(sell_layout(blen.p, (int)nC, SELL_SIGMA, bmap, bpos, bsp, &nb, &bt, s));
            // B^T: the pairs, and behind them the single unknowns, are sorted by length within
            // windows where their own order pads much (a pair then takes the longer of its rows
            // twice, so what stays is at most about twice the entries)
            ASSS_TRY(pair_layout(tlen.p, nuslots, tsp, &tt, s));
            if ((double)tt > SELL_PAD * (double)nt) {
                DBuf<int> plen, slen, back, pmap, smap;
                ASSS_TRY(plen.alloc(npairs));
                ASSS_TRY(slen.alloc(nsingle));
                k_pair_len<<<cdiv(npairs + nsingle, 256), 256, 0, s>>>((int)npairs, (int)nsingle, tlen.p, plen.p, slen.p);
                ASSS_CHECK_LAUNCH();
                ASSS_TRY(sort_windows(plen.p, (int)npairs, SELL_SIGMA, back, pmap, s));
                ASSS_TRY(sort_windows(slen.p, (int)nsingle, SELL_SIGMA, back, smap, s));
                ASSS_TRY(place(pmap.p, smap.p));
                ASSS_TRY(pair_layout(tlen.p, nuslots, tsp, &tt, s));   // (synchronises: the maps are freed here)
            }
        }
        if (bsp.p && tsp.p && 12.0 * (double)(bt + tt) + vectors <= budget) {
            DBuf<int> bcol, tcol, its_d;
            DBuf<double> bval, tval, m1, m2, sv, zz, pp, qq, rr, part, rel_d;
            DBuf<unsigned> bar;
            DBuf<int> err;
            ASSS_TRY(bcol.alloc(bt > 0 ? bt : 1));
            ASSS_TRY(bval.alloc(bt > 0 ? bt : 1));
            ASSS_TRY(tcol.alloc(tt > 0 ? tt : 1));
            ASSS_TRY(tval.alloc(tt > 0 ? tt : 1));
            for (DBuf<double>* v : {&m1, &m2, &sv, &zz, &pp}) ASSS_TRY(v->alloc(nuslots));
            ASSS_TRY(qq.alloc(32LL * nbs));
            ASSS_TRY(rr.alloc(32LL * nbs));
            k_bx_fill<<<cdiv(32LL * nbs, 256), 256, 0, s>>>(32 * nbs, (int)nC, bmap.p, klist.p, prow.p, P.ci.p, Abar.rp.p,
                                                             Abar.ci.p, Abar.v.p, ST.rp.p, ST.ci.p, st_src.p, upos.p, sg,
                                                             bsp.p, bcol.p, bval.p, rr.p);
            ASSS_CHECK_LAUNCH();
            k_btx_fill<<<cdiv(nuslots, 256), 256, 0, s>>>(nuslots, uslot.p, srow.p, Spat.ci.p, AbarT.rp.p, AbarT.ci.p,
                                                           AbarT.v.p, P.rp.p, P.ci.p, mirror.p, cidx.p, bpos.p, sg, tsp.p,
                                                           tcol.p, tval.p, Nn.p, partner.p, cross.p, s0, m1.p, m2.p, sv.p);
            ASSS_CHECK_LAUNCH();
            int occ = 0;
            ASSS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_lls_pcg, PCG_THREADS, 0));
            if (occ < 1) {
                set_error("least-squares kernel cannot be resident");
                return ASSS_ERR_CUDA;
            }
            int nblk = c.sms * (occ > 2 ? 2 : occ);
            const int want = cdiv(nbs > nts ? nbs : nts, PCG_THREADS / 32);
            if (nblk > want) nblk = want > 0 ? want : 1;
            ASSS_TRY(part.alloc(4LL * nblk));
            ASSS_TRY(bar.alloc(1));
            ASSS_TRY(err.alloc(1));
            ASSS_TRY(its_d.alloc(1));
            ASSS_TRY(rel_d.alloc(1));
            ASSS_CUDA(cudaMemsetAsync(bar.p, 0, sizeof(unsigned), s));
            ASSS_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), s));
            PcgParams a;
            a.nb = nbs;
            a.nt = nts;
            a.bsp = bsp.p;
            a.bcol = bcol.p;
            a.tsp = tsp.p;
            a.tcol = tcol.p;
            a.bval = bval.p;
            a.tval = tval.p;
            a.m1 = m1.p;
            a.m2 = m2.p;
            a.q = qq.p;
            a.rho = rr.p;
            a.p = pp.p;
            a.z = zz.p;
            a.s = sv.p;
            a.part = part.p;
            a.gb.count = bar.p;
            a.gb.err = err.p;
            a.budget = c.wait_cycles;
            a.tol = tol;
            a.maxit = maxit;
            a.has_s0 = s0 != nullptr;
            a.cs = stream_evict_first(c, 12 * (bt + tt)) ? 1 : 0;
            a.its = its_d.p;
            a.rel = rel_d.p;
            void* args[] = {&a};
            ASSS_CUDA(cudaLaunchCooperativeKernel((const void*)k_lls_pcg, dim3(nblk), dim3(PCG_THREADS), args, 0, s));
            count_launch();
            ASSS_TRY(s_val.alloc(nS));
            k_unslot<<<cdiv(nS, 256), 256, 0, s>>>(nS, upos.p, sv.p, s_val.p);
            ASSS_CHECK_LAUNCH();
            ASSS_TRY(Cval.alloc(nP));
            ASSS_TRY(lls_product_on_pattern(c, Abar, ST, st_src.p, s_val.p, P, prow.p, Cval.p));
            int hi = 0, he = 0;
            double hr = 0.0;
            ASSS_CUDA(cudaMemcpyAsync(&he, err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
            ASSS_CUDA(cudaMemcpyAsync(&hi, its_d.p, sizeof(int), cudaMemcpyDeviceToHost, s));
            ASSS_CUDA(cudaMemcpyAsync(&hr, rel_d.p, sizeof(double), cudaMemcpyDeviceToHost, s));
            ASSS_CUDA(cudaStreamSynchronize(s));
            if (he) {
                set_error("least-squares fit: a grid barrier wait exceeded its budget");
                return (asss_status)he;
            }
            if (res) {
                res->its = hi;
                res->relgrad = hr;
            }
            return ASSS_OK;
        }
    }
    // ---- matrix-free ----
    DBuf<double> rho, q, r, z, p, sc;
    ASSS_TRY(s_val.alloc(nS));
    ASSS_TRY(rho.alloc(nP));
    ASSS_TRY(q.alloc(nP));
    ASSS_TRY(r.alloc(nS));
    ASSS_TRY(z.alloc(nS));
    ASSS_TRY(p.alloc(nS));
    ASSS_TRY(sc.alloc(8));  // 0: rz, 1: qq, 2: rr, 3: rz_new, 4: rr0
    double* d_rz = sc.p;
    double* d_qq = sc.p + 1;
    double* d_rr = sc.p + 2;
    double* d_rzn = sc.p + 3;
    ASSS_CUDA(cudaMemsetAsync(s_val.p, 0, sizeof(double) * nS, s));
    k_lls_init_rho<<<cdiv(nP, 256), 256, 0, s>>>(nP, prow.p, P.ci.p, sg, rho.p);
    ASSS_CHECK_LAUNCH();
    auto applyBT = [&](const double* t, double* g) -> asss_status {
        k_lls_BT<<<cdiv(nS, 256), 256, 0, s>>>(nS, srow.p, Spat.ci.p, AbarT.rp.p, AbarT.ci.p, AbarT.v.p, P.rp.p, P.ci.p,
                                                mirror.p, t, sg, g);
        ASSS_CHECK_LAUNCH();
        return ASSS_OK;
    };
    auto applyB = [&](const double* sv, double* out) -> asss_status {
        k_lls_B<<<cdiv(nP, 256), 256, 0, s>>>(nP, prow.p, P.ci.p, Abar.rp.p, Abar.ci.p, Abar.v.p, ST.rp.p, ST.ci.p,
                                               st_src.p, sv, sg, out);
        ASSS_CHECK_LAUNCH();
        return ASSS_OK;
    };
    auto precond = [&]() -> asss_status {
        k_lls_prec_apply<<<cdiv(nS, 256), 256, 0, s>>>(nS, Nn.p, partner.p, cross.p, r.p, z.p);
        ASSS_CHECK_LAUNCH();
        return ASSS_OK;
    };
    // the tolerance is relative to ||B^T v|| (the gradient at s = 0), also when the
    // iteration starts from given values s0 (a set-up resumed from saved S values)
    ASSS_TRY(applyBT(rho.p, r.p));
    ASSS_TRY(dot(r.p, r.p, nS, d_rr, s));
    double rr0 = 0.0;
    ASSS_CUDA(cudaMemcpyAsync(&rr0, d_rr, sizeof(double), cudaMemcpyDeviceToHost, s));
    ASSS_CUDA(cudaStreamSynchronize(s));
    double rel = rr0 > 0 ? 1.0 : 0.0;
    if (s0 && rr0 > 0) {
        ASSS_CUDA(cudaMemcpyAsync(s_val.p, s0, sizeof(double) * nS, cudaMemcpyDeviceToDevice, s));
        ASSS_TRY(applyB(s_val.p, q.p));
        ASSS_TRY(vaxpy(rho.p, q.p, -1.0, nP, s));  // rho = v - B s0
        ASSS_TRY(applyBT(rho.p, r.p));
        ASSS_TRY(dot(r.p, r.p, nS, d_rr, s));
        double rr = 0.0;
        ASSS_CUDA(cudaMemcpyAsync(&rr, d_rr, sizeof(double), cudaMemcpyDeviceToHost, s));
        ASSS_CUDA(cudaStreamSynchronize(s));
        rel = sqrt(rr / rr0);
    }
    ASSS_TRY(precond());
    ASSS_TRY(vcopy(p.p, z.p, nS, s));
    ASSS_TRY(dot(r.p, z.p, nS, d_rz, s));
    int its = 0;
    const int check_every = 8;
    int mx = nS > nP ? nS : nP;
    while (rr0 > 0 && rel > tol && its < maxit) {
        ASSS_TRY(applyB(p.p, q.p));
        ASSS_TRY(dot(q.p, q.p, nP, d_qq, s));
        k_cg_update<<<cdiv(mx, 256), 256, 0, s>>>(s_val.p, p.p, nS, rho.p, q.p, nP, d_rz, d_qq);
        ASSS_CHECK_LAUNCH();
        ASSS_TRY(applyBT(rho.p, r.p));
        ASSS_TRY(precond());
        ASSS_TRY(dot(r.p, z.p, nS, d_rzn, s));
        k_cg_newp<<<cdiv(nS, 256), 256, 0, s>>>(p.p, z.p, nS, d_rzn, d_rz);
        ASSS_CHECK_LAUNCH();
        ASSS_CUDA(cudaMemcpyAsync(d_rz, d_rzn, sizeof(double), cudaMemcpyDeviceToDevice, s));
        ++its;
        if (its % check_every == 0 || its == maxit) {
            ASSS_TRY(dot(r.p, r.p, nS, d_rr, s));
            double rr = 0.0;
            ASSS_CUDA(cudaMemcpyAsync(&rr, d_rr, sizeof(double), cudaMemcpyDeviceToHost, s));
            ASSS_CUDA(cudaStreamSynchronize(s));
            rel = sqrt(rr / rr0);
            if (rel <= tol) break;
        }
    }
    if (res) {
        res->its = its;
        res->relgrad = rel;
    }
    ASSS_TRY(Cval.alloc(nP));
    ASSS_TRY(lls_product_on_pattern(c, Abar, ST, st_src.p, s_val.p, P, prow.p, Cval.p));
    return ASSS_OK;
}

}  // namespace asss
