// dp_ref.cu -- fp64 reference kernels of the approximate DP (Sec. 5) and the
// traceback / evaluation that every DP pass ends with.
//
// The reference DP evaluates every candidate of eq. apx_rec in binary64 with
// interval costs from double-double prefix differences (App. E), one layer per
// launch.  It is the slow, exact path (ECASQ_DP_REFERENCE) against which the
// fast kernel is validated; the traceback and evaluation kernels serve both.
#include "common.cuh"

namespace ecasq {

void timer_begin(cudaStream_t st);
void timer_end(cudaStream_t st);

struct Lams { double v[kMaxG]; };

__device__ __forceinline__ size_t dp_at(int g, int i, int64_t j, int s, int64_t p) {
    return ((size_t)g * (size_t)(s + 1) + (size_t)i) * (size_t)p + (size_t)j;
}

// Rows 0, 1 and every undefined entry: dp = +inf, bp = -1.
__global__ void k_dp_clear(double *dp64, int32_t *bp, int G, int s, int64_t p) {
    size_t n = (size_t)G * (size_t)(s + 1) * (size_t)p;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) { dp64[i] = CUDART_INF; bp[i] = -1; }
}

// eq. apx_base: dp(2, j) = min over a in L, a < j, of C[a, j] + lambda' Phi^first[a, j]
// (lowest a among exact minima; L = {0} when P = X).
__global__ void k_dp_base(Prefix P, Lams lam, int G, int s, double *dp64, int32_t *bp) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1;
    if (j >= P.p) return;
    double best[kMaxG];
    int32_t arg[kMaxG];
#pragma unroll
    for (int g = 0; g < kMaxG; g++) { best[g] = CUDART_INF; arg[g] = -1; }
    for (int64_t a = 0; a < P.nL && a < j; a++) {
        double C, U, D;
        pair_exact(P, a, j, C, U, D);
        double phi = phi_first_at(P, a, U, D);
#pragma unroll
        for (int g = 0; g < kMaxG; g++) {
            if (g < G) {
                double c = __dadd_rn(C, __dmul_rn(lam.v[g], phi));
                if (c < best[g]) { best[g] = c; arg[g] = (int32_t)a; }
            }
        }
    }
    for (int g = 0; g < G; g++) {
        dp64[dp_at(g, 2, j, s, P.ps)] = best[g];
        bp[dp_at(g, 2, j, s, P.ps)] = arg[g];
    }
}

// eq. apx_rec, one layer i >= 3 for all G multipliers: thread per j, every
// k in [i-2, j-1], candidate dp(i-1, k) + (C[k,j] + lambda' Phi[k,j]); the
// lowest k among exact minima wins.  Heavy (large-j) blocks launch first.
__global__ void __launch_bounds__(128) k_dp_layer_ref(Prefix P, Lams lam, int G, int s, int i, double *dp64,
                                                      int32_t *bp) {
    int64_t nblk = gridDim.x;
    int64_t j = (nblk - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
    if (j < i - 1 || j >= P.p) return;
    double best[kMaxG];
    int32_t arg[kMaxG];
#pragma unroll
    for (int g = 0; g < kMaxG; g++) { best[g] = CUDART_INF; arg[g] = -1; }
    for (int64_t k = i - 2; k < j; k++) {
        double C, U, D;
        pair_exact(P, k, j, C, U, D);
        double phi = phi_exact(P, U, D, false);
#pragma unroll
        for (int g = 0; g < kMaxG; g++) {
            if (g < G) {
                double prev = dp64[dp_at(g, i - 1, k, s, P.ps)];
                double c = __dadd_rn(prev, __dadd_rn(C, __dmul_rn(lam.v[g], phi)));
                if (c < best[g]) { best[g] = c; arg[g] = (int32_t)k; }
            }
        }
    }
    for (int g = 0; g < G; g++) {
        dp64[dp_at(g, i, j, s, P.ps)] = best[g];
        bp[dp_at(g, i, j, s, P.ps)] = arg[g];
    }
}

// eq. apx_final over i and j in R (smallest i, then smallest j, among exact minima;
// i = s only with EXACT_S) and the backpointer walk down to the first value
// a = bp(2, .), then the metrics of the traced codebook.  Block g = one multiplier,
// one warp.
__global__ void k_traceback_eval(Prefix P, int G, int s, int exact_s, const double *dp64, const int32_t *bp,
                                 int32_t *qidx, int32_t *mcount, double *metrics) {
    __shared__ double scratch[4 * kMaxS];
    __shared__ int32_t a[kMaxS];
    __shared__ int sm_m;
    int g = blockIdx.x;
    int64_t p = P.p;
    // eq. apx_final over the lanes: the least value, the first (i, then j) among equal ones
    const int ilo = exact_s ? s : 2;
    const int64_t last = (int64_t)(s - ilo + 1) * P.nR;
    double best = CUDART_INF;
    int64_t first = last;
    for (int64_t q = threadIdx.x; q < last; q += 32) {
        const double v = dp64[dp_at(g, ilo + (int)(q / P.nR), p - P.nR + q % P.nR, s, P.ps)];
        if (v < best) { best = v; first = q; }
    }
    for (int o = 16; o; o >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, best, o);
        const int64_t q = __shfl_xor_sync(0xffffffffu, first, o);
        const long long k = order_key(v), k0 = order_key(best);
        if (q < last && (first == last || k < k0 || (k == k0 && q < first))) { best = v; first = q; }
    }
    if (threadIdx.x == 0) {
        const int istar = first < last ? ilo + (int)(first / P.nR) : -1;
        const int64_t jstar = first < last ? p - P.nR + first % P.nR : -1;
        if (istar < 0) {
            sm_m = 0;
        } else {
            int64_t j = jstar;
            a[istar - 1] = (int32_t)j;
            bool ok = true;  // every output on the path carries a backpointer (not so after a timed-out wait)
            for (int i = istar; i >= 3 && ok; i--) {
                j = bp[dp_at(g, i, j, s, P.ps)];
                ok = j >= 0;
                a[i - 2] = (int32_t)j;
            }
            if (ok) a[0] = bp[dp_at(g, 2, j, s, P.ps)];
            sm_m = (ok && a[0] >= 0) ? istar : 0;
        }
        metrics[4 * g + 0] = best;
        mcount[g] = sm_m;
    }
    __syncwarp();
    int m = sm_m;
    for (int r = threadIdx.x; r < m; r += 32) qidx[g * s + r] = a[r];
    if (m > 0 && m <= 32)
        eval_codebook_lanes(P, a, m, &metrics[4 * g + 1]);  // the same values, one interval per lane
    else if (m > 0)
        eval_codebook_warp(P, a, m, &metrics[4 * g + 1], scratch);
}

// Metrics of a caller-given codebook (unique indices on the device); nothing when
// gate is given and holds 0 (the caller then reads no result).
__global__ void k_eval_codebook(Prefix P, const int32_t *a_in, int m, double *out3, const int32_t *gate) {
    __shared__ double scratch[4 * kMaxS];
    __shared__ int32_t a[kMaxS];
    if (gate && *gate == 0) return;
    for (int r = threadIdx.x; r < m; r += 32) a[r] = a_in[r];
    __syncwarp();
    if (m <= 32)
        eval_codebook_lanes(P, a, m, out3);  // the same values, one interval per lane
    else
        eval_codebook_warp(P, a, m, out3, scratch);
}

// Q[r] = v[a[r]] for every multiplier row g.
__global__ void k_gather_q(const float *v, const int32_t *qidx, const int32_t *mcount, int s, float *Q) {
    int g = blockIdx.x;
    int m = mcount[g];
    for (int r = threadIdx.x; r < m; r += blockDim.x) Q[g * s + r] = v[qidx[g * s + r]];
}

// Unique indices of a codebook given by value (binary search in v); -1 if absent.
__global__ void k_locate_q(const float *v, int64_t p, const float *Q, int m, int32_t *a, DevStatus *st) {
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        float q = Q[r];
        if (q == 0.0f) q = 0.0f;
        int64_t lo = 0, hi = p - 1;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (v[mid] < q) lo = mid + 1; else hi = mid;
        }
        bool ok = v[lo] == q;
        a[r] = ok ? (int32_t)lo : -1;
        if (!ok) st->range_err = 1;
    }
}

// ----------------------------------------------------------- host launchers
// Tables cleared (dp = +inf, bp = -1) and layer 2 (eq. apx_base) filled.
int launch_dp_clear_base(const Prefix &P, const double *lamp, int G, int s, double *dp64, int32_t *bp,
                         cudaStream_t st) {
    Lams lam{};
    for (int g = 0; g < G; g++) lam.v[g] = lamp[g];
    note_launch();
    k_dp_clear<<<4096, 256, 0, st>>>(dp64, bp, G, s, P.ps);
    ECASQ_LAUNCH_CHECK();
    if (P.p >= 2) {
        note_launch();
        // (a warp a block: its binary64 sequence is 5 us of an SM's pipe)
        k_dp_base<<<(unsigned)cdiv(P.p - 1, 32), 32, 0, st>>>(P, lam, G, s, dp64, bp);
        ECASQ_LAUNCH_CHECK();
    }
    return ECASQ_OK;
}

int launch_dp_reference(const Prefix &P, const double *lamp, int G, int s, double *dp64, int32_t *bp,
                        cudaStream_t st) {
    Lams lam{};
    for (int g = 0; g < G; g++) lam.v[g] = lamp[g];
    int rc = launch_dp_clear_base(P, lamp, G, s, dp64, bp, st);
    if (rc != ECASQ_OK) return rc;
    timer_begin(st);
    for (int i = 3; i <= s; i++) {
        if (P.p < i) break;
        note_launch();
        k_dp_layer_ref<<<(unsigned)cdiv(P.p, 128), 128, 0, st>>>(P, lam, G, s, i, dp64, bp);
        ECASQ_LAUNCH_CHECK();
    }
    timer_end(st);
    return ECASQ_OK;
}

int launch_traceback_eval(const Prefix &P, int G, int s, int exact_s, const double *dp64, const int32_t *bp,
                          int32_t *qidx, int32_t *mcount, double *metrics, cudaStream_t st) {
    note_launch();
    k_traceback_eval<<<G, 32, 0, st>>>(P, G, s, exact_s, dp64, bp, qidx, mcount, metrics);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

int launch_eval_codebook(const Prefix &P, const int32_t *a, int m, double *out3, cudaStream_t st,
                         const int32_t *gate) {
    note_launch();
    k_eval_codebook<<<1, 32, 0, st>>>(P, a, m, out3, gate);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

int launch_gather_q(const float *v, const int32_t *qidx, const int32_t *mcount, int G, int s, float *Q,
                    cudaStream_t st) {
    note_launch();
    k_gather_q<<<G, 64, 0, st>>>(v, qidx, mcount, s, Q);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

int launch_locate_q(const float *v, int64_t p, const float *Q, int m, int32_t *a, DevStatus *ds, cudaStream_t st) {
    note_launch();
    k_locate_q<<<1, 256, 0, st>>>(v, p, Q, m, a, ds);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

}  // namespace ecasq
