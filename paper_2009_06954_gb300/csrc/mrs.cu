// Host side of the persistent mrs solve (mrs_kernel.cuh): the workspace, the choice of
// the operator's storage, the deferred statistics, and the allocation-free entry point.
#include "mrs_kernel.cuh"

namespace asss {

asss_status mrs_work_create(MrsWork** w, int n, int sms) {
    MrsWork* m = new MrsWork();
    m->n = n;
    m->sms = sms;
    asss_status st = ASSS_OK;
    int maxblk = sms * 4;
    if ((st = m->part.alloc((int64_t)2 * (MRS_KPMAX + 1) * maxblk)) != ASSS_OK ||
        (st = m->bar.alloc(2)) != ASSS_OK || (st = m->err.alloc(1)) != ASSS_OK ||
        (st = m->out_its.alloc(1)) != ASSS_OK || (st = m->out_ratio.alloc(1)) != ASSS_OK ||
        (st = m->blk_slice.alloc(maxblk + 1)) != ASSS_OK) {
        delete m;
        return st;
    }
    if (cudaEventCreate(&m->ev0) != cudaSuccess || cudaEventCreate(&m->ev1) != cudaSuccess) {
        delete m;
        set_error("cudaEventCreate failed");
        return ASSS_ERR_CUDA;
    }
    if (getenv("ASSS_TRACE_MRS") && (st = m->trace.alloc(MRS_TRACE_SLOTS)) != ASSS_OK) {
        delete m;
        return st;
    }
    if ((st = m->its_log.alloc(MrsWork::LOG_CAP)) != ASSS_OK ||
        (st = m->ratio_log.alloc(MrsWork::LOG_CAP)) != ASSS_OK) {
        delete m;
        return st;
    }
    if (cudaMemset(m->err.p, 0, sizeof(int)) != cudaSuccess) {
        delete m;
        set_error("cudaMemset failed");
        return ASSS_ERR_CUDA;
    }
    *w = m;
    return ASSS_OK;
}

void mrs_work_destroy(MrsWork* w) { delete w; }

// Y ring with zero halos of width H on both ends of each slot (re-zeroed whenever
// the layout changes; the kernel never writes the halos)
template <class T>
static asss_status y_layout(MrsWork* w, DBuf<T>& Ybuf, int& cur, int H, cudaStream_t s, T** Y, long long* ystride) {
    H = (int)pad32(H);   // every slot's row 0 starts on 128 bytes
    const long long st = pad32(w->n) + 2LL * H;
    if (cur != H || Ybuf.n < 3 * st) {
        if (Ybuf.n < 3 * st) ASSS_TRY(Ybuf.alloc(3 * st));
        ASSS_CUDA(cudaMemsetAsync(Ybuf.p, 0, sizeof(T) * (size_t)Ybuf.n, s));
        cur = H;
    }
    *Y = Ybuf.p + H;
    *ystride = st;
    return ASSS_OK;
}

template <class T>
static asss_status dispatch_mrs(const Ctx& c, MrsWork* w, const DSell<T>* sell, const DSkewDia<T>* dia, const T* Q,
                                const double* alpha, int k, int kp, double shift, double sign, const double* rhs,
                                T* x, DBuf<T>& Ybuf, int& ylay, T* P, double tol, int maxit, long long* nnz_read,
                                LaunchOut lo, const __nv_bfloat16* Q16 = nullptr, int kp16 = 0,
                                const IldlFactor* fac = nullptr, const DStream<T>* rows = nullptr) {
    OpView<T> v;
    if (dia && dia->ndiag > MRS_MAXDIAG) dia = nullptr;
    T* Y = nullptr;
    long long ystride = 0;
    ASSS_TRY(y_layout<T>(w, Ybuf, ylay, (dia && !fac) ? dia->halo : 0, c.stream, &Y, &ystride));
    if (fac) {
        if (Q16) {
            set_error("the factored inner operator reads Q_k in FP32 or FP64 only");
            return ASSS_ERR_UNSUPPORTED;
        }
        v.n = fac->n;
        v.fmt = 3;
        v.nslices = cdiv(fac->n, 32);
        v.key = fac;
        v.fac = fac;
        v.nnz = fac->nl + fac->nu + fac->nj;
        *nnz_read = v.nnz;
        return dispatch_kp<T, 3>(c, w, v, Q, alpha, k, kp, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
    }
    if (dia) {
        v.n = dia->n;
        v.fmt = 1;
        v.nslices = cdiv(dia->n, 32);
        v.ndiag = dia->ndiag;
        v.off = dia->off.p;
        v.U = dia->U.p + dia->halo;
        v.ustride = dia->ustride;
        v.halo = dia->halo;
        v.key = dia;
        v.nnz = dia->nnz;
        *nnz_read = v.nnz;
        if constexpr (sizeof(T) == 4) {
            if (Q16) return dispatch_kp16<1>(c, w, v, Q16, alpha, k, kp16, shift, sign, rhs, x, Y, ystride, P, tol,
                                             maxit, lo);
        }
        if constexpr (sizeof(T) == 8) {
            // at most a slice per SM: four lanes a row
            if (v.nslices <= c.sms) {
                v.fmt = 5;
                return dispatch_kp<T, 5>(c, w, v, Q, alpha, k, kp, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
            }
        }
        return dispatch_kp<T, 1>(c, w, v, Q, alpha, k, kp, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
    }
    if (rows) {
        v.n = rows->n;
        v.fmt = 4;
        v.nslices = cdiv(rows->n, 32);
        v.rrp = rows->rp.p;
        v.rcol = rows->col.p;
        v.rval = rows->val.p;
        v.rstored = rows->nstored;
        v.key = rows;
        v.nnz = rows->nnz;
        *nnz_read = v.nnz;
        if constexpr (sizeof(T) == 4) {
            if (Q16) return dispatch_kp16<4>(c, w, v, Q16, alpha, k, kp16, shift, sign, rhs, x, Y, ystride, P, tol,
                                             maxit, lo);
        }
        return dispatch_kp<T, 4>(c, w, v, Q, alpha, k, kp, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
    }
    if (!sell) {
        set_error("mrs: no operator storage");
        return ASSS_ERR_ARG;
    }
    v.n = sell->n;
    v.fmt = 0;
    v.nslices = sell->nslices;
    v.sptr = sell->sptr.p;
    v.col = sell->col.p;
    v.val = sell->val.p;
    v.rowmap = sell->rowmap.p;
    v.units = sell->units.p;
    v.uoff = sell->uoff.p;
    v.hacc = const_cast<T*>(sell->hacc.p);
    v.hcnt = const_cast<unsigned*>(sell->hcnt.p);
    v.nheavy = sell->nheavy;
    v.split = sell->split;
    v.key = sell;
    v.nnz = sell->nnz;
    *nnz_read = v.nnz;
    if constexpr (sizeof(T) == 4) {
        if (Q16) return dispatch_kp16<0>(c, w, v, Q16, alpha, k, kp16, shift, sign, rhs, x, Y, ystride, P, tol, maxit,
                                         lo);
    }
    return dispatch_kp<T, 0>(c, w, v, Q, alpha, k, kp, shift, sign, rhs, x, Y, ystride, P, tol, maxit, lo);
}

asss_status mrs_solve(const Ctx& c, MrsWork* w, const MrsOperator& op, bool fp32, double shift, double sign,
                      const double* rhs, double* x64, float* x32, double tol, int maxit, double* qtz, MrsResult* res,
                      bool sync_result) {
    NvtxRange nv_("asss:mrs");
    int n = w->n;
    if (w->log_n == MrsWork::LOG_CAP) ASSS_TRY(mrs_collect(c, w, nullptr));
    LaunchOut lo{w->log_n, qtz};
    while ((int)w->evs.size() < 2 * (lo.slot + 1)) {
        cudaEvent_t e;
        ASSS_CUDA(cudaEventCreate(&e));
        w->evs.push_back(e);
    }
    long long nnz_read = 0;
    if (fp32) {
        if ((!op.J32 && !op.D32 && !op.F && !op.R32) || !x32) {
            set_error("FP32 mrs needs the FP32 operator and an FP32 output");
            return ASSS_ERR_ARG;
        }
        if (!w->P32.p) ASSS_TRY(w->P32.alloc(2 * pad32(n)));
        ASSS_TRY(dispatch_mrs<float>(c, w, op.J32, op.D32, op.Q32, op.alpha, op.k, op.kp, shift, sign, rhs, x32,
                                     w->Y32, w->halo32, w->P32.p, tol, maxit, &nnz_read, lo,
                                     (const __nv_bfloat16*)op.Q16, op.kp16, op.F, op.R32));
    } else {
        if ((!op.J64 && !op.D64 && !op.F && !op.R64) || !x64) {
            set_error("FP64 mrs needs the FP64 operator and an FP64 output");
            return ASSS_ERR_ARG;
        }
        if (!w->P64.p) ASSS_TRY(w->P64.alloc(2 * pad32(n)));
        ASSS_TRY(dispatch_mrs<double>(c, w, op.J64, op.D64, op.Q64, op.alpha, op.k, op.kp, shift, sign, rhs, x64,
                                      w->Y64, w->halo64, w->P64.p, tol, maxit, &nnz_read, lo, nullptr, 0, op.F,
                                      op.R64));
    }
    // algorithmic bytes: set-up pass (rhs in FP64, Y/x/P written, Q row), per step
    // (matrix entries - SELL ones with a 4-byte index -, Q row, gathered/own y,
    // y_old, y_new, p r/w, x r/w), final pass (y, p, x r/w; Q^T x needs no pass over Q)
    long long T = fp32 ? 4 : 8;
    long long nn = n, kp = op.kp;
    long long qrow = (fp32 && op.Q16) ? 2LL * op.kp16 : kp * T;  // bytes of one Q row as read
    const bool dia = !op.F && (fp32 ? op.D32 != nullptr : op.D64 != nullptr);
    const bool rows = !op.F && !dia && (fp32 ? op.R32 != nullptr : op.R64 != nullptr);
    const long long per_entry = dia ? T : rows ? T + 2 : T + 4;   // SELL: 32-bit columns; row stream: 16-bit
    if ((int)w->log_nnz.size() <= lo.slot) {
        w->log_nnz.resize(lo.slot + 1);
        w->log_per_row.resize(lo.slot + 1);
    }
    w->log_nnz[lo.slot] = nn * (8 + 4 * T + qrow) + nn * 4 * T;
    // factored operator: + wd, t written and gathered, w written and gathered, per step
    w->log_per_row[lo.slot] = nnz_read * per_entry + nn * (7 * T + qrow) + (op.F ? nn * 5 * T : 0);
    w->log_n++;
    if (sync_result) {
        std::vector<MrsResult> v;
        ASSS_TRY(mrs_collect(c, w, &v));
        if (res) *res = v.back();
    }
    return ASSS_OK;
}

asss_status mrs_collect(const Ctx& c, MrsWork* w, std::vector<MrsResult>* out) {
    int nl = w->log_n;
    if (nl == 0) return ASSS_OK;
    std::vector<int> its(nl);
    std::vector<double> ratio(nl);
    int herr = 0;
    ASSS_CUDA(cudaMemcpyAsync(its.data(), w->its_log.p, sizeof(int) * nl, cudaMemcpyDeviceToHost, c.stream));
    ASSS_CUDA(cudaMemcpyAsync(ratio.data(), w->ratio_log.p, sizeof(double) * nl, cudaMemcpyDeviceToHost, c.stream));
    ASSS_CUDA(cudaMemcpyAsync(&herr, w->err.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    std::vector<unsigned long long> tl(w->trace.p ? MRS_TRACE_SLOTS : 0);
    if (w->trace.p)
        ASSS_CUDA(cudaMemcpyAsync(tl.data(), w->trace.p, sizeof(unsigned long long) * MRS_TRACE_SLOTS,
                                  cudaMemcpyDeviceToHost, c.stream));
    ASSS_CUDA(cudaStreamSynchronize(c.stream));
    w->log_n = 0;
    if (w->trace.p) {
        // last launch: phase durations in ns (block 0)
        fprintf(stderr, "mrs timeline (block 0, ns): phase0-pass %llu barrier %llu setup %llu |",
                tl[1] - tl[0], tl[2] - tl[1], tl[3] - tl[2]);
        int steps = its[nl - 1] < MRS_TRACE_STEPS ? its[nl - 1] : MRS_TRACE_STEPS;
        for (int j = 1; j < steps; ++j) {
            int tb = 4 + 5 * (j - 1);
            unsigned long long prev = (j == 1) ? tl[3] : tl[tb - 1];
            fprintf(stderr, " [pass %llu part %llu bar %llu red %llu sc+u %llu]", tl[tb] - prev,
                    tl[tb + 1] - tl[tb], tl[tb + 2] - tl[tb + 1], tl[tb + 3] - tl[tb + 2], tl[tb + 4] - tl[tb + 3]);
        }
        fprintf(stderr, "\n");
    }
    for (int i = 0; i < nl; ++i) {
        if (its[i] < 0) continue;  // a launch that found its skip flag set did no work
        float ms = 0.f;
        ASSS_CUDA(cudaEventElapsedTime(&ms, w->evs[2 * i], w->evs[2 * i + 1]));
        MrsResult r;
        r.its = its[i];
        r.ratio = ratio[i];
        r.status = herr;
        r.ms = ms;
        r.bytes = w->log_nnz[i] + (long long)its[i] * w->log_per_row[i];
        w->tot.its += r.its;
        w->tot.launches += 1;
        w->tot.ms += r.ms;
        w->tot.bytes += r.bytes;
        if (out) out->push_back(r);
    }
    if (herr) {
        // the status word is sticky until read here: later launches exit at once
        ASSS_CUDA(cudaMemsetAsync(w->err.p, 0, sizeof(int), c.stream));
        set_error("mrs: a grid barrier wait exceeded its budget");
        return (asss_status)herr;
    }
    return ASSS_OK;
}

void mrs_set_skip(MrsWork* w, const int* flag) { w->skip = flag; }
const int* mrs_get_skip(const MrsWork* w) { return w->skip; }

MrsTotals mrs_take_totals(MrsWork* w) {
    MrsTotals t = w->tot;
    w->tot = MrsTotals();
    return t;
}


// ===========================================================================
// Allocation-free entry point.  Its scratch is one file-scope device array, so
// the call itself never allocates device memory.
// ===========================================================================
constexpr long long NOALLOC_MAX_N = 1LL << 16;
constexpr int NOALLOC_MAX_BLOCKS = 512;
constexpr long long NOALLOC_CTRL = 8;                                          // control words
constexpr long long NOALLOC_PART = 2LL * (MRS_KPMAX + 1) * NOALLOC_MAX_BLOCKS;  // reduction partials
constexpr long long NOALLOC_BLK = (NOALLOC_MAX_BLOCKS + 2) / 2;                // block->slice table (ints)
constexpr long long NOALLOC_DOUBLES = NOALLOC_CTRL + NOALLOC_PART + NOALLOC_BLK + 5 * NOALLOC_MAX_N;

// [ctrl | partials | block table | Y: 3 slots of n | P: 2 slots of n]
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_DOUBLES];

static double* noalloc_base(int* status) {
    static std::mutex mu;
    static double* base[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 256) {
        set_error("cudaGetDevice failed: %s", cudaGetErrorString(e));
        *status = ASSS_ERR_CUDA;
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (!base[dev]) {
        double* ptr = nullptr;
        e = cudaGetSymbolAddress((void**)&ptr, g_noalloc_scratch);
        if (e != cudaSuccess || !ptr) {
            set_error("cudaGetSymbolAddress of the static scratch failed: %s", cudaGetErrorString(e));
            *status = ASSS_ERR_CUDA;
            return nullptr;
        }
        base[dev] = ptr;
    }
    *status = ASSS_OK;
    return base[dev];
}

__global__ void k_noalloc_check_rp(const int64_t* rp, int64_t n, int64_t nnz, int* flag) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n) return;
    int64_t v = rp[i];
    if ((i == 0 && v != 0) || (i == n && v != nnz) || v < 0 || v > nnz || (i < n && rp[i + 1] < v)) atomicOr(flag, 1);
}

__global__ void k_noalloc_check_ci(const int64_t* rp, const int32_t* ci, int64_t n, int* flag) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e)
        if (ci[e] < 0 || ci[e] >= n) {
            atomicOr(flag, 2);
            return;
        }
}

// columns k..kp-1 of the row-major q must be zero: they enter x through q[m] * u[m]
// with u[m] = 0, so a NaN or Inf there would turn x into NaN
__global__ void k_noalloc_check_qpad(const double* q, int64_t n, int k, int kp, int* flag) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int w = kp - k;
    if (w <= 0 || t >= n * w) return;
    const int64_t i = t / w;
    const int m = k + (int)(t % w);
    if (q[i * kp + m] != 0.0) atomicOr(flag, 4);
}

template <int KP>
static asss_status noalloc_launch(int nblk, cudaStream_t s, MrsParams<double>& prm) {
    void* args[] = {&prm};
    ASSS_CUDA(cudaLaunchCooperativeKernel((const void*)k_mrs<double, KP, 2>, dim3(nblk),
                                          dim3(mrs_threads<double, 2>()), args, 0, s));
    count_launch();
    return ASSS_OK;
}

template <int KP>
static asss_status noalloc_occupancy(int* occ) {
    ASSS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_mrs<double, KP, 2>, (mrs_threads<double, 2>()), 0));
    return ASSS_OK;
}

}  // namespace asss

using namespace asss;

extern "C" asss_status asss_mrs_noalloc(int64_t n, int64_t nnz, const int64_t* row_ptr, const int32_t* col_idx,
                                        const double* val, int k, int kp, const double* q_rowmajor,
                                        const double* alpha, double shift, double sign, const double* b, double* x,
                                        double tol, int maxit, int* its, double* ratio, void* stream) {
    if (n < 1 || n > NOALLOC_MAX_N) {
        set_error("asss_mrs_noalloc: n = %lld is outside 1..%lld, the size of its static scratch", (long long)n,
                  NOALLOC_MAX_N);
        return ASSS_ERR_ARG;
    }
    if (nnz < 0 || nnz >= (1LL << 40) || !row_ptr || !col_idx || !val || !b || !x || maxit < 1 || !(shift > 0.0) ||
        k < 0 || k > kp ||
        (k > 0 && !q_rowmajor) || (k > 1 && !alpha)) {
        set_error("asss_mrs_noalloc: invalid arguments");
        return ASSS_ERR_ARG;
    }
    if (sign != 1.0 && sign != -1.0) {
        set_error("asss_mrs_noalloc: sign must be +1 or -1");
        return ASSS_ERR_ARG;
    }
    int cur_dev = 0;
    ASSS_CUDA(cudaGetDevice(&cur_dev));
    // every array is read in place by the kernel: it must be memory of the current
    // device (another GPU's memory would be read without peer access) and aligned for
    // the kernel's vector loads (q rows are read 16 bytes at a time)
    struct Arr {
        const void* p;
        size_t align;
        const char* name;
    };
    const Arr arrs[] = {{row_ptr, 8, "row_ptr"}, {col_idx, 4, "col_idx"}, {val, 8, "val"},
                        {b, 8, "b"},             {x, 8, "x"},             {k > 0 ? q_rowmajor : nullptr, 16, "q"},
                        {k > 1 ? alpha : nullptr, 8, "alpha"}};
    for (const Arr& a : arrs) {
        if (!a.p) continue;
        if (ptr_place(a.p, cur_dev) != PtrPlace::HERE) {
            set_error("asss_mrs_noalloc: %s must be device memory of the current device %d", a.name, cur_dev);
            return ASSS_ERR_ARG;
        }
        if (((uintptr_t)a.p) % a.align != 0) {
            set_error("asss_mrs_noalloc: %s must be aligned to %zu bytes", a.name, a.align);
            return ASSS_ERR_ARG;
        }
    }
    int st = ASSS_OK;
    double* base = noalloc_base(&st);
    if (!base) return (asss_status)st;
    cudaStream_t s = (cudaStream_t)stream;
    Ctx c;
    ASSS_TRY(make_ctx(c, stream, 2000.0));
    int occ = 0;
    switch (kp) {
#define NA_OCC(KPV) \
    case KPV:       \
        ASSS_TRY(noalloc_occupancy<KPV>(&occ)); \
        break;
        NA_OCC(0) NA_OCC(4) NA_OCC(8) NA_OCC(12) NA_OCC(16) NA_OCC(20) NA_OCC(24) NA_OCC(32) NA_OCC(48) NA_OCC(64)
#undef NA_OCC
        default:
            set_error("asss_mrs_noalloc: kp must be one of 0,4,8,12,16,20,24,32,48,64");
            return ASSS_ERR_ARG;
    }
    if (occ < 1) {
        set_error("mrs kernel cannot be resident");
        return ASSS_ERR_CUDA;
    }
    int nslices = (int)((n + 31) / 32);
    int nblk = mrs_blocks<double, 2>(c.sms, occ, nslices);
    if (nblk > NOALLOC_MAX_BLOCKS) nblk = NOALLOC_MAX_BLOCKS;
    unsigned* ctrl = reinterpret_cast<unsigned*>(base);  // [0] count [2] err [3] its; ratio at base[3]
    double* part = base + NOALLOC_CTRL;
    int* blk = reinterpret_cast<int*>(base + NOALLOC_CTRL + NOALLOC_PART);
    double* Y = base + NOALLOC_CTRL + NOALLOC_PART + NOALLOC_BLK;
    double* P = Y + 3 * n;
    // the control words must start at zero; everything else is written before it is read
    ASSS_CUDA(cudaMemsetAsync(base, 0, sizeof(double) * NOALLOC_CTRL, s));
    // the CSR is read in place: check row pointers, then column indices (flag in ctrl[2])
    {
        int* flag = reinterpret_cast<int*>(ctrl + 2);
        k_noalloc_check_rp<<<(int)((n + 256) / 256), 256, 0, s>>>(row_ptr, n, nnz, flag);
        ASSS_CHECK_LAUNCH();
        int hf = 0;
        ASSS_CUDA(cudaMemcpyAsync(&hf, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
        ASSS_CUDA(cudaStreamSynchronize(s));
        if (!hf) {
            k_noalloc_check_ci<<<(int)((n + 255) / 256), 256, 0, s>>>(row_ptr, col_idx, n, flag);
            ASSS_CHECK_LAUNCH();
            if (k > 0 && kp > k) {
                const int64_t cnt = n * (int64_t)(kp - k);
                k_noalloc_check_qpad<<<(int)((cnt + 255) / 256), 256, 0, s>>>(q_rowmajor, n, k, kp, flag);
                ASSS_CHECK_LAUNCH();
            }
            ASSS_CUDA(cudaMemcpyAsync(&hf, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
            ASSS_CUDA(cudaStreamSynchronize(s));
        }
        if (hf & 3) {
            set_error("asss_mrs_noalloc: malformed CSR (row pointers or column indices)");
            return ASSS_ERR_PATTERN;
        }
        if (hf) {
            set_error("asss_mrs_noalloc: columns k..kp-1 of q must be zero");
            return ASSS_ERR_ARG;
        }
    }
    k_partition<<<(nblk + 128) / 128, 128, 0, s>>>(nullptr, nslices, nblk, blk);
    ASSS_CHECK_LAUNCH();
    MrsParams<double> prm;
    memset(&prm, 0, sizeof(prm));
    prm.n = (int)n;
    prm.crp = (const long long*)row_ptr;
    prm.cci = col_idx;
    prm.cval = val;
    prm.ystride = n;
    prm.pstride = n;
    prm.Q = q_rowmajor;
    prm.alpha = alpha;
    prm.k = k;
    prm.shift = shift;
    prm.sign = sign;
    prm.rhs = b;
    prm.x = x;
    prm.Y = Y;
    prm.P = P;
    prm.part = part;
    prm.gb.count = ctrl;
    prm.gb.err = reinterpret_cast<int*>(ctrl + 2);
    prm.blk_slice = blk;
    prm.tol = tol;
    prm.maxit = maxit;
    prm.budget = c.wait_cycles;
    prm.out_its = reinterpret_cast<int*>(ctrl + 3);
    prm.out_ratio = base + 3;
    prm.qtz = nullptr;
    switch (kp) {
#define NA_CASE(KPV) \
    case KPV:        \
        ASSS_TRY(noalloc_launch<KPV>(nblk, s, prm)); \
        break;
        NA_CASE(0) NA_CASE(4) NA_CASE(8) NA_CASE(12) NA_CASE(16) NA_CASE(20) NA_CASE(24) NA_CASE(32) NA_CASE(48)
        NA_CASE(64)
#undef NA_CASE
    }
    unsigned h[4] = {0, 0, 0, 0};
    double hr = 0.0;
    ASSS_CUDA(cudaMemcpyAsync(h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, s));
    ASSS_CUDA(cudaMemcpyAsync(&hr, base + 3, sizeof(double), cudaMemcpyDeviceToHost, s));
    ASSS_CUDA(cudaStreamSynchronize(s));
    if (h[2]) {
        set_error("asss_mrs_noalloc: a grid barrier wait exceeded its budget");
        return ASSS_ERR_TIMEOUT;
    }
    if (its) *its = (int)h[3];
    if (ratio) *ratio = hr;
    return ASSS_OK;
}
