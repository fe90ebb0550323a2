// The small levels' V-cycle as one explicit matrix.
//
// With the dense coarsest solve the V-cycle from any level l down is a fixed
// linear operator x_l = B_l b_l (arxiv 2210.16660, Sec. 3.1, Eq.
// (multiplicative composition)), symmetric for the l1-Jacobi and for the
// forward/backward Gauss-Seidel smoother. On the smallest levels applying its
// levels one by one is a chain of short dependent steps (levels of 4,073 rows
// and less of the 64^3 mesh: 21 us in one thread-block cluster), while B_l of
// up to kOpRows rows is one matrix-vector product (1,036 rows: 8.6 MB read
// from L2). Setup and refresh form B_l from the finished levels in float64:
// one block per column runs the V-cycle's step at level l on a unit vector,
// with B_{l+1} (the coarsest inverse at the end) as its coarse correction.
// Every entry is formed and applied in float64 in either V-cycle precision.
#include <cstdio>

#include "internal.cuh"

namespace pcgamg {
namespace {

constexpr int kOpThreads = 256;
// Largest level applied as a matrix. The product is bounded by the float64
// pipe (n^2 FMAs at 304 a clock: 1,036 rows 1.7 us), two more sweeps and a
// smaller matrix by latency (about 2 us each). Alone, 400 rows instead cost
// 812 us per 24^3 solve (834-row level, 727 with it), 1,536 and 2,600 rows the
// same there, but 128^3 22.9 ms with 2,600 (22.0); 41^3 float64 (a level between
// 1,100 and 1,280 rows) 2,412 us without it, 2,230 with it. Systems that share
// the pipe would rather have less: twelve at once 12.6 ms with 1,280, 12.5 with
// 900 and 13.2 with 1,536, 48 of 24^3 to 112^3 198.7 and 196.6 with 900, where
// the same 48 one by one take 272 either way (277 with 600, 282 with 300).
constexpr int kOpRows = 1280;

// One level's step, for column j (blockIdx.x) of B: x = S e_j + correction,
// the smoothing and transfer steps of the V-cycle in plain float64.
struct OpLevel {
    int n, nc;
    const int32_t *rp, *ci;
    const double *v, *dinv;
    const int32_t *agg, *rptr, *ridx;                 // tentative transfers
    const double *p;
    const int32_t *prp, *pci, *trp, *tci;             // smoothed transfers (P, P^T), or null
    const double *pv, *tv;
    const double *Bc;                                 // nc x nc
    int nu, nb;                                       // Gauss-Seidel sweeps and rows per block; nu = 0: l1-Jacobi
    double *B;                                        // n x n
};

// One Gauss-Seidel sweep (see k_gs_sweep) of x_old into x_new, b = e_j.
template <bool FWD>
__device__ void op_sweep(const OpLevel &a, int j, const double *xo, double *xn, bool zero) {
    for (int64_t lo64 = (int64_t)threadIdx.x * a.nb; lo64 < a.n; lo64 += (int64_t)blockDim.x * a.nb) {
        const int lo = (int)lo64, hi = (int)min((int64_t)a.n, lo64 + a.nb);
        for (int r = lo; r < hi; r++) xn[r] = zero ? 0.0 : xo[r];
        for (int q = 0; q < hi - lo; q++) {
            const int r = FWD ? lo + q : hi - 1 - q;
            double acc = 0.0;
            for (int32_t k = a.rp[r]; k < a.rp[r + 1]; k++) {
                const int c = a.ci[k];
                acc += a.v[k] * (c >= lo && c < hi ? xn[c] : (zero ? 0.0 : xo[c]));
            }
            xn[r] += a.dinv[r] * ((r == j ? 1.0 : 0.0) - acc);
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kOpThreads) k_op_column(OpLevel a) {
    extern __shared__ double sm[];
    const int n = a.n, nc = a.nc, j = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    double *x = sm, *y = sm + n, *r = sm + 2 * n, *rc = sm + 3 * n, *xc = rc + nc;
    // pre-smoothing from zero
    if (a.nu == 0) {
        for (int i = tid; i < n; i += nt) x[i] = i == j ? a.dinv[i] : 0.0;
        __syncthreads();
    } else {
        for (int sw = 0; sw < a.nu; sw++) {
            op_sweep<true>(a, j, x, y, sw == 0);
            double *t = x;
            x = y;
            y = t;
        }
    }
    // residual and restriction
    for (int i = tid; i < n; i += nt) {
        double acc = 0.0;
        for (int32_t k = a.rp[i]; k < a.rp[i + 1]; k++) acc += a.v[k] * x[a.ci[k]];
        r[i] = (i == j ? 1.0 : 0.0) - acc;
    }
    __syncthreads();
    for (int I = tid; I < nc; I += nt) {
        double s = 0.0;
        if (a.prp) {
            for (int32_t q = a.trp[I]; q < a.trp[I + 1]; q++) s += a.tv[q] * r[a.tci[q]];
        } else {
            for (int32_t q = a.rptr[I]; q < a.rptr[I + 1]; q++) s += a.p[a.ridx[q]] * r[a.ridx[q]];
        }
        rc[I] = s;
    }
    __syncthreads();
    // coarse correction (Bc is symmetric: read by columns, coalesced)
    for (int I = tid; I < nc; I += nt) {
        double s = 0.0;
        for (int J = 0; J < nc; J++) s += a.Bc[(int64_t)J * nc + I] * rc[J];
        xc[I] = s;
    }
    __syncthreads();
    for (int i = tid; i < n; i += nt) {
        if (a.prp) {
            double s = 0.0;
            for (int32_t q = a.prp[i]; q < a.prp[i + 1]; q++) s += a.pv[q] * xc[a.pci[q]];
            x[i] += s;
        } else if (a.agg[i] >= 0) {
            x[i] += a.p[i] * xc[a.agg[i]];
        }
    }
    __syncthreads();
    // post-smoothing
    if (a.nu == 0) {
        for (int i = tid; i < n; i += nt) {
            double acc = 0.0;
            for (int32_t k = a.rp[i]; k < a.rp[i + 1]; k++) acc += a.v[k] * x[a.ci[k]];
            a.B[(int64_t)i * n + j] = x[i] + a.dinv[i] * ((i == j ? 1.0 : 0.0) - acc);
        }
        return;
    }
    for (int sw = 0; sw < a.nu; sw++) {
        op_sweep<false>(a, j, x, y, false);
        double *t = x;
        x = y;
        y = t;
    }
    for (int i = tid; i < n; i += nt) a.B[(int64_t)i * n + j] = x[i];
}

}  // namespace

// Picks op_first and allocates the matrices: the first level >= 1 of at most
// kOpRows rows, or the coarsest one (whose matrix is there already). They may
// take what dropping the int32 columns has given back, or any free memory of a
// handle without a budget; when they do not fit, op_first stays 0 and the
// small levels run as before.
int ops_alloc(amg_hier *h) {
    Mem &M = h->mem;
    const int L = (int)h->lev.size() - 1;
    h->op_first = 0;
    h->op.assign(L + 1, nullptr);
    if (h->coarse_iter || L == 0 || h->no_op) return AMG_OK;
    int D = 1;
    while (D < L && h->lev[D].A.n > kOpRows) D++;
    size_t need = 0;
    for (int l = D; l < L; l++) need += sizeof(double) * (size_t)h->lev[l].A.n * h->lev[l].A.n + 256;
    if (M.budget && D < L && need > h->col_bytes) return AMG_OK;
    for (int l = D; l < L; l++) {
        const size_t n = h->lev[l].A.n;
        if (alloc(M, &h->op[l], n * n)) {
            cudaGetLastError();
            set_error("");
            for (double *&q : h->op) release(M, q);
            return AMG_OK;
        }
    }
    if (h->lev[D].A.n > h->nL) {
        release(M, h->bL);
        PCG_TRY(alloc(M, &h->bL, h->lev[D].A.n));
    }
    h->op_first = D;
    return AMG_OK;
}

// Forms op[l] for l = L-1..op_first from the levels' current values, for the
// smoother (nu, nblocks) of amg_set_smoother.
int ops_build(amg_hier *h, int nu, int nblocks, cudaStream_t s) {
    const int L = (int)h->lev.size() - 1;
    if (!h->op_first) return AMG_OK;
    for (int l = L - 1; l >= h->op_first; l--) {
        Level &lv = h->lev[l];
        OpLevel a = {};
        a.n = lv.A.n;
        a.nc = h->lev[l + 1].A.n;
        a.rp = lv.A.rp;
        a.ci = lv.A.ci;
        a.v = lv.A.v;
        a.dinv = lv.dinv;
        a.agg = lv.agg;
        a.rptr = lv.rptr;
        a.ridx = lv.ridx;
        a.p = lv.p;
        if (h->smoothed) {
            a.prp = lv.P.rp;
            a.pci = lv.P.ci;
            a.pv = lv.P.v;
            a.trp = lv.Pt.rp;
            a.tci = lv.Pt.ci;
            a.tv = lv.Pt.v;
        }
        a.Bc = l + 1 == L ? h->Ainv : h->op[l + 1];
        a.nu = nu;
        a.nb = nu > 0 ? gs_rows(lv.A.n, nblocks) : 1;
        a.B = h->op[l];
        const size_t smem = sizeof(double) * (3 * (size_t)a.n + 2 * (size_t)a.nc);
        PCG_CK(cudaFuncSetAttribute(k_op_column, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(5 * kOpRows * sizeof(double))));
        k_op_column<<<a.n, kOpThreads, smem, s>>>(a);
        PCG_LAUNCH_CK();
    }
    return AMG_OK;
}

}  // namespace pcgamg
