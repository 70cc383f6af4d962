// rows.cu -- one DP pass of the multiplier search for many independent rows of at most kScanTile
// values (Sec. 5, eqs. apx_base / apx_rec / apx_final), a block per row, all layers in one launch.
//
// The pass needs a codebook and its metrics per multiplier, so only decisions have to be exact:
//  1. k_rows_build, once per search: the fp32 interval costs C, Phi of every pair k < j (cost32.cuh:
//     one column a thread, k descending from the empty interval; a row is short enough that the
//     compensated sums need no anchors: n^2 u^2 <= 2^-28) and the binary64 base costs C[0, j],
//     Phi^first[0, j].  The row is scaled by a power of two that brings its largest magnitude
//     into [2^30, 2^31), or lower where a multiplier of the first pass is beyond 2^118 then, so that
//     neither the costs nor lambda' overflow and two values at least 2^-100 apart keep the relative bounds.
//     A row with a smaller gap, or one below 2^-70 of its largest magnitude (an interval of that length has its
//     Phi only as well as double-double sums have its mean), takes its binary64 costs rounded; one whose binary64
//     costs are not costs (a mean outside its interval, an entropy below zero), or a later multiplier beyond
//     2^120, is left to the caller (mcount = -1).
//  2. k_rows_pass: eq. apx_rec in fp32, layer by layer, eight multipliers at a time.
//  3. The traceback, a warp per multiplier.  At an output the candidates within the certified band
//     of the fp32 minimum hold the exact minimiser; where it is the only one, the decision is exact.
//     Elsewhere, and between last layers, the members' closure is evaluated in binary64 with
//     double-double interval costs (resolve; lowest k, smallest i among exact minima).
// The results are those of the binary64 recurrence: every output's candidate set is that of the
// fast DP (dp_fast.cu), and an exact minimum of one candidate needs no evaluation.  The bound that this rests on is
// checked at run time, as there: an output resolved, those of its closure where that is large, and every
// codebook's objective from its binary64 metrics have to lie within the certified error of their fp32
// values (row_within; counted in DevStatus::bound_viol).
//
// What bounds it: the chip has 2 binary64 operations a cycle and SM, so an interval cost for every pair
// (8128 a row of 128 values) took 43 of 70 ms of device time for 8192 rows at s = 8; fp32 costs
// and binary64 only for ambiguous decisions and the metrics take 10 (0.5 for the costs, 1.6 a round);
// 64 rows of 300 values at s = 8: 1.1 ms of device time instead of 64 single solves of 3.6 ms.  The second bound was the
// scan of one output a thread with a marker bit per candidate (2 candidates a cycle and SM); here a
// unit (32 columns, 16 or 32 k) loads a pair's costs once for eight multipliers.
#include <algorithm>

#include "common.cuh"
#include "cost32.cuh"

namespace ecasq {

constexpr int kRowsThreads = 512;   // at most; 256 for rows whose costs fit shared memory
constexpr float kRowsMinGap = 0x1p-100f;

// Pair (k, j) of a row at pair_at(k, j, p): k-major, so the lanes of a warp (consecutive j, one k) touch
// consecutive words.
__device__ __forceinline__ int pair_at(int k, int j, int p) { return k * p - k * (k + 1) / 2 + j - k - 1; }
// The row's scale exponent for multipliers up to lam: the largest magnitude is v[0]'s or v[p-1]'s.
__device__ __forceinline__ int row_exp(const float *v, int p, double lam) {
    const int e = 30 - ilogbf(fmaxf(fabsf(v[0]), fabsf(v[p - 1])));
    return lam > 0.0 ? min(e, (117 - ilogb(lam)) >> 1) : e;
}

__device__ __forceinline__ Prefix row_prefix(const RowsData &R, int64_t row, int p) {
    Prefix P;
    P.v = R.v + row * R.dcap;
    P.w = R.w + row * R.dcap;
    P.N = R.N + row * (R.dcap + 1);
    P.S = R.S + row * 2 * (R.dcap + 1);
    P.S2 = R.S2 + row * 2 * (R.dcap + 1);
    P.p = p;
    P.d = R.d;
    P.ps = p;
    return P;
}

// A row's kept costs: fp32 {C, Phi} by pair, then C[0, j] and Phi^first[0, j].  Phi^first[0, 0] (unused) is its costs' scale, C[0, 0]
// (unused) the noise that row_within allows a layer, or -1 for a row that fp32 cannot take.
struct RowCosts { float2 *cf; double *c0, *phf; };
__device__ __forceinline__ RowCosts row_costs(const RowsPass &A, int64_t row) {
    double *g = A.pairs + row * A.pstride;
    double *c0 = g + (A.pstride - 2 * A.R.dcap);
    return {reinterpret_cast<float2 *>(g), c0, c0 + A.R.dcap};
}

// The binary64 costs of a row's pairs, rounded (2 binary64 operations a cycle and SM: a search of 512 rows of 128 values takes
// 5.3 ms instead of 2.1).  C below zero is within the run-time check's noise of it.  Returns whether this thread met what is
// no cost.
static __device__ __noinline__ bool rows_build_rounded(const Prefix &P, const RowCosts &rc, double scale) {
    const int p = (int)P.p;
    bool lost = false;
    for (int j = threadIdx.x; j < p; j += blockDim.x)
        for (int k = 0; k < j; k++) {
            double C, U, D;
            pair_exact(P, k, j, C, U, D);
            if (k == 0) {
                rc.c0[j] = C;
                const double F = phi_exact(P, U, D, true);
                rc.phf[j] = F;
                lost |= !(F >= 0.0);
            }
            const double F = phi_exact(P, U, D, false);
            rc.cf[pair_at(k, j, p)] = make_float2(fmaxf(__double2float_rn(__dmul_rn(C, scale)), 0.f) + 0.f,
                                                  __double2float_rn(F) + 0.f);
            lost |= !(F >= 0.0);
        }
    return lost;
}

__global__ void __launch_bounds__(kScanTile) k_rows_build(const RowsPass A) {
    __shared__ float v[kScanTile], w[kScanTile];
    const int64_t row = A.rows[blockIdx.x];
    const int p = (int)A.R.p[row];
    const Prefix P = row_prefix(A.R, row, p);
    const RowCosts rc = row_costs(A, row);
    double lmax = 0.0;
#pragma unroll
    for (int g = 0; g < kMaxG; g++)  // (as integers: multipliers are >= 0)
        lmax = __longlong_as_double(max(__double_as_longlong(lmax), __double_as_longlong(g < A.G ? A.lam[(size_t)blockIdx.x * A.G + g] : 0.0)));
    const int e = row_exp(P.v, p, lmax);
    for (int t = threadIdx.x; t < p; t += blockDim.x) {
        v[t] = ldexpf(P.v[t], e);
        w[t] = (float)P.w[t];
    }
    __syncthreads();
    const float gap = fmaxf(kRowsMinGap, 0x1p-70f * fmaxf(fabsf(v[0]), fabsf(v[p - 1])));
    bool narrow = false;
    for (int t = threadIdx.x; t + 1 < p; t += blockDim.x) narrow |= !(__fsub_rn(v[t + 1], v[t]) >= gap);
    narrow = __syncthreads_or(narrow);
    bool lost = false;
    if (narrow) lost = __syncthreads_or(rows_build_rounded(P, rc, ldexp(1.0, 2 * e)));
    if (threadIdx.x == 0) {
        rc.phf[0] = ldexp(1.0, 2 * e);
        rc.c0[0] = lost ? -1.0 : ldexp(A.R.norm2[row], 2 * e - 90);
    }
    if (narrow) return;
    const float d_f = (float)P.d, invd = 1.0f / (float)P.d;
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x; j - lane < p; j += blockDim.x) {
        const int jt = j - lane;  // the warp's first column
        const float vj = v[min(j, p - 1)];
        Rec r = rec_empty();
        for (int k = min(jt + 30, p - 2); k >= 0; k--) {
            if (k < j && j < p) {
                rec_step(r, vj, v[k + 1], w[k + 1], __fsub_rn(v[k + 1], v[k]));
                float2 c;
                rec_emit(r, vj, v[k], d_f, invd, c.x, c.y);
                rc.cf[pair_at(k, j, p)] = c;
            }
        }
        if (j >= 1 && j < p) {
            double C, U, D;
            pair_exact(P, 0, j, C, U, D);
            rc.c0[j] = C;
            rc.phf[j] = phi_exact(P, U, D, true);
        }
    }
}

// What a warp knows of its multiplier while it traces and resolves.
struct RowTrace {
    Prefix P;
    const float2 *cf;
    const double *c0, *phf;
    const float *dp;       // [s+1][p][8] fp32
    double *dp64;          // [s+1][p]: exact values of the closure's outputs
    uint16_t *list;        // [s+1][p]: the closure's outputs by layer
    uint32_t *need;        // [s+1][nw]: ... as bits, all zero between traces
    uint16_t *arg;         // [s+1][p]: ... their lowest minimisers
    uint16_t *cnt, *from;  // [s+1]: ... their number by layer; before the present closure
    uint32_t *key;         // [kRowsPairs]: pairs to evaluate
    double *cost;          // [kRowsPairs]: ... and their costs
    const float *tau;
    double lam, scale;
    float lam32, slack, noise;
    int p, g, nw;
    int *tally;            // outputs outside their certified error, candidates evaluated (shared memory)
};
__device__ __forceinline__ float row_limit(const RowTrace &T, int i, float m) {
    return __fadd_ru(__fmul_ru(m, __fadd_ru(1.0f, T.tau[i])), T.slack);
}
// Whether the fp32 value m32 of an output of layer i is within its certified error of the exact one, best * scale: eps_i
// and 2^-24 for the rounding of `best`, as the comparison is fp32 (tau_i / 2 is above both; layer 2 has no band), the
// underflow that row_limit allows for, and what double-double interval costs and their sums leave, `noise` a layer: 2^-100 of
// N V^2 <= 2^10 ||X||^2 (V the largest magnitude).
__device__ __forceinline__ bool row_within(float m32, double best, float tau, float slack, double scale, int i, float noise) {
    const float x = __double2float_rn(__dmul_rn(best, scale));
    return fabsf(m32 - x) <= (i > 2 ? 0.5f * tau : 0x1.001p-23f) * x + (slack + (float)i * noise);
}
// Members of output (i, j) among k = kb .. kb + 127, 32 a word: candidates whose fp32 value (the forward pass's) is not
// above the limit.  One warp; the loads of the four words are in flight together.
__device__ __forceinline__ void row_members(const RowTrace &T, int i, int j, int kb, float lim, unsigned (&in)[4]) {
    const int lane = threadIdx.x & 31;
    float d[4];
    float2 c[4];
#pragma unroll
    for (int w = 0; w < 4; w++) {
        const int k = kb + 32 * w + lane;
        d[w] = CUDART_INF_F;
        c[w] = make_float2(0.f, 0.f);
        if (k < j) {
            d[w] = T.dp[((size_t)(i - 1) * T.p + k) * kMaxG + T.g];
            c[w] = T.cf[pair_at(k, j, T.p)];
        }
    }
#pragma unroll
    for (int w = 0; w < 4; w++) {
        const float v = __fadd_rn(d[w], __fmaf_rn(T.lam32, c[w].y, c[w].x));
        in[w] = __ballot_sync(0xffffffffu, kb + 32 * w + lane < j && !(v > lim));
    }
}
__device__ __forceinline__ double row_base(const RowTrace &T, int j) {
    return __dadd_rn(T.c0[j], __dmul_rn(T.lam, T.phf[j]));
}

// Binary64 candidate cost C[k, j] + lambda' Phi[k, j].
__device__ __forceinline__ double row_cost(const RowTrace &T, int k, int j) {
    double C, U, D;
    pair_exact(T.P, k, j, C, U, D);
    return __dadd_rn(C, __dmul_rn(T.lam, phi_exact(T.P, U, D, false)));
}

__device__ __forceinline__ int row_outside(const RowTrace &T, int i, int j, double best) {
    return row_within(T.dp[((size_t)i * T.p + j) * kMaxG + T.g], best, T.tau[i], T.slack, T.scale, i, T.noise) ? 0 : 1;
}

// Whether output (i, j) is listed, and so resolved once its closure is.
__device__ __forceinline__ bool row_listed(const RowTrace &T, int i, int j) {
    return (T.need[(size_t)i * T.nw + (j >> 5)] >> (j & 31)) & 1u;
}
// Lists the outputs kb + bits of `any` of layer i that are not listed yet, behind the n that are; their number then.
__device__ __forceinline__ int row_list(const RowTrace &T, int i, int kb, unsigned any, int n) {
    const int lane = threadIdx.x & 31;
    uint32_t *word = T.need + (size_t)i * T.nw + (kb >> 5);
    const unsigned old = *word, fresh = any & ~old;
    __syncwarp();
    if (lane == 0) *word = old | any;
    if ((fresh >> lane) & 1u) T.list[(size_t)i * T.p + n + __popc(fresh & ((1u << lane) - 1u))] = (uint16_t)(kb + lane);
    return n + __popc(fresh);
}
// row_members for 32 outputs of layer i at once, a lane one: members among k = kb .. kb + 31 of output j.
__device__ __forceinline__ unsigned row_members_of(const RowTrace &T, int i, int j, int kb, float lim) {
    unsigned in = 0u;
    const float *d = T.dp + ((size_t)(i - 1) * T.p + kb) * kMaxG + T.g;
    const float2 *cp = T.cf + pair_at(kb, j, T.p);
#pragma unroll 8
    for (int t = 0; t < 32; t++) {
        const int k = kb + t;
        float v = CUDART_INF_F;
        if (k < j) {
            const float2 c = *cp;
            v = __fadd_rn(d[t * kMaxG], __fmaf_rn(T.lam32, c.y, c.x));
        }
        cp += T.p - k - 2;  // the next k's row starts one pair later
        if (k < j && !(v > lim)) in |= 1u << t;
    }
    return in;
}
constexpr int kRowsPairs = 64;  // costs that are evaluated side by side (RowsPass::cost: 64 costs, 64 keys)
constexpr int kRowsWide = 8;    // outputs of a layer from which a lane takes one

// Candidates T.key[at .. at + n - 1] (j << 10 | k) of layer i, n <= 32, a lane one: into their outputs' least value and
// lowest minimiser.
__device__ __forceinline__ void row_evaluate_pairs(const RowTrace &T, int i, int at, int n) {
    const int lane = threadIdx.x & 31, p = T.p;
    const unsigned full = 0xffffffffu;
    const bool have = lane < n;
    const uint32_t f = have ? T.key[at + lane] : 0u;
    int k = (int)(f & 1023u);
    const int j = have ? (int)(f >> 10) : -1 - lane;
    double c = CUDART_INF;
    if (have) c = __dadd_rn(i == 3 ? row_base(T, k) : T.dp64[(size_t)(i - 1) * p + k], row_cost(T, k, j));
    const unsigned peers = __match_any_sync(full, j);
    const bool leader = have && lane == __ffs(peers) - 1;
    for (unsigned rest = __ballot_sync(full, leader && (peers & (peers - 1u))); rest; rest &= rest - 1u) {
        const int l = __ffs(rest) - 1;
        const bool mine = (__shfl_sync(full, peers, l) >> lane) & 1u;
        const long long own = mine ? order_key(c) : 0x7fffffffffffffffll;
        long long x = own;
        int y = mine ? k : 0x7fffffff;
        for (int o = 16; o; o >>= 1) {
            const long long x2 = __shfl_xor_sync(full, x, o);
            const int y2 = __shfl_xor_sync(full, y, o);
            if (x2 < x || (x2 == x && y2 < y)) { x = x2; y = y2; }
        }
        const double least = __shfl_sync(full, c, __ffs(__ballot_sync(full, mine && own == x && k == y)) - 1);
        if (lane == l) { c = least; k = y; }
    }
    if (leader) {
        const size_t o = (size_t)i * p + j;
        const long long x = order_key(c), y = order_key(T.dp64[o]);
        if (x < y || (x == y && k < (int)T.arg[o])) { T.dp64[o] = c; T.arg[o] = (uint16_t)k; }
    }
    __syncwarp();
}

// The listed outputs of a large closure from layer 3 up, those behind `from` in each layer's list: members are found again and
// queued, 32 candidates at a time evaluated side by side, whatever outputs they are of.
static __device__ __noinline__ void row_resolve_many(const RowTrace &T, int i0) {
    const int lane = threadIdx.x & 31, p = T.p;
    const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
    int bad = 0;
    for (int i = 3; i <= i0; i++) {
        const int n0 = T.from[i], n1 = T.cnt[i];
        const uint16_t *list = T.list + (size_t)i * p;
        for (int e = n0 + lane; e < n1; e += 32) {
            T.dp64[(size_t)i * p + list[e]] = CUDART_INF;
            T.arg[(size_t)i * p + list[e]] = 0xFFFFu;
        }
        __syncwarp();
        int qn = 0;
        auto queue = [&](bool in, int j, int k) {  // whole warp
            const unsigned m = __ballot_sync(full, in);
            if (in) T.key[qn + __popc(m & lt)] = (uint32_t)(j << 10 | k);
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) row_evaluate_pairs(T, i, qn -= 32, 32);
        };
        if (n1 - n0 >= kRowsWide) {
            for (int b = n0; b < n1; b += 32) {
                const int j = b + lane < n1 ? (int)list[b + lane] : 0, jmax = __reduce_max_sync(full, j);
                const float lim = row_limit(T, i, T.dp[((size_t)i * p + j) * kMaxG + T.g]);
                for (int kb = 0; kb < jmax; kb += 32) {
                    unsigned in = row_members_of(T, i, j, kb, lim);
                    while (__any_sync(full, in)) {
                        queue(in != 0u, j, kb + __ffs(in) - 1);
                        in &= in - 1u;
                    }
                }
            }
        } else {
            for (int e = n0; e < n1; e++) {
                const int j = list[e];
                const float lim = row_limit(T, i, T.dp[((size_t)i * p + j) * kMaxG + T.g]);
                for (int kb = 0; kb < j; kb += 128) {
                    unsigned in[4];
                    row_members(T, i, j, kb, lim, in);
#pragma unroll 1
                    for (int w = 0; w < 4; w++) {
                        const unsigned x = w == 0 ? in[0] : w == 1 ? in[1] : w == 2 ? in[2] : in[3];
                        if (x) queue((x >> lane) & 1u, j, kb + 32 * w + lane);
                    }
                }
            }
        }
        if (qn) row_evaluate_pairs(T, i, 0, qn);
        for (int e = n0 + lane; e < n1; e += 32) bad += row_outside(T, i, list[e], T.dp64[(size_t)i * p + list[e]]);
    }
    if (bad) atomicAdd(T.tally, bad);
    __syncwarp();
}

// The exact value and lowest minimiser of output (i0, j0), i0 >= 3: its members, their members and so on
// down to layer 3 are listed (each output once a trace), then evaluated from layer 3 up.  One warp.  A binary64 interval
// cost is a long chain whose time 32 lanes share, so up to kRowsPairs costs of the closure (nearly
// always all) are evaluated side by side first; larger closures -- evenly spaced values tie in thousands of
// outputs -- layer by layer (row_resolve_many).  What was resolved stays known until the trace ends (dp64, arg), so
// that a trace evaluates an output once and follows the rest of its path (row_follow): 4 rows of 107 integers at s = 64 took 261 ms output by output
// and closure by closure, and take 4.3 (5.0 with every pair's binary64 cost kept).
// known: the trace has resolved outputs.
static __device__ __noinline__ int row_resolve(const RowTrace &T, int i0, int j0, bool known, double *value) {
    const int lane = threadIdx.x & 31, p = T.p;
    const unsigned full = 0xffffffffu;
    uint16_t *cnt = T.cnt;
    if (known && row_listed(T, i0, j0)) {
        *value = T.dp64[(size_t)i0 * p + j0];
        return T.arg[(size_t)i0 * p + j0];
    }
    for (int i = 3 + lane; i <= i0; i += 32) T.from[i] = cnt[i];
    __syncwarp();
    if (lane == 0) {
        atomicOr(&T.need[(size_t)i0 * T.nw + (j0 >> 5)], 1u << (j0 & 31));
        T.list[(size_t)i0 * p + cnt[i0]++] = (uint16_t)j0;
    }
    __syncwarp();
    int np = 0;
    bool wide = false;
    for (int i = i0; i >= 3; i--) {
        const int n0 = T.from[i], n1 = cnt[i];
        if (n0 == n1) continue;
        int nn = i > 3 ? cnt[i - 1] : 0;
        if (n1 - n0 >= kRowsWide) {
            wide = true;
            for (int b = n0; b < n1; b += 32) {
                const int j = b + lane < n1 ? (int)T.list[(size_t)i * p + b + lane] : 0, jmax = __reduce_max_sync(full, j);
                const float lim = row_limit(T, i, T.dp[((size_t)i * p + j) * kMaxG + T.g]);
                for (int kb = 0; kb < jmax; kb += 32) {
                    const unsigned in = row_members_of(T, i, j, kb, lim), any = __reduce_or_sync(full, in);
                    np += __reduce_add_sync(full, __popc(in));
                    if (any && i > 3) nn = row_list(T, i - 1, kb, any, nn);
                    __syncwarp();
                }
            }
        } else {
            for (int e = n0; e < n1; e++) {
                const int j = T.list[(size_t)i * p + e];
                const float lim = row_limit(T, i, T.dp[((size_t)i * p + j) * kMaxG + T.g]);
                for (int kb = 0; kb < j; kb += 128) {
                    unsigned in[4];
                    row_members(T, i, j, kb, lim, in);
#pragma unroll
                    for (int w = 0; w < 4; w++) {
                        if (!in[w]) continue;
                        const int k = kb + 32 * w + lane, q = np + __popc(in[w] & ((1u << lane) - 1u));
                        if (((in[w] >> lane) & 1u) && q < kRowsPairs) T.key[q] = (uint32_t)(i << 20 | j << 10 | k);
                        np += __popc(in[w]);
                        if (i > 3) nn = row_list(T, i - 1, kb + 32 * w, in[w], nn);
                        __syncwarp();
                    }
                }
            }
        }
        if (lane == 0 && i > 3) cnt[i - 1] = (uint16_t)nn;
        __syncwarp();
    }
    if (lane == 0) atomicAdd(T.tally + 1, np);
    if (wide || np > kRowsPairs) {
        row_resolve_many(T, i0);
        *value = T.dp64[(size_t)i0 * p + j0];
        return T.arg[(size_t)i0 * p + j0];
    }
    for (int q = lane; q < np; q += 32) T.cost[q] = row_cost(T, (int)(T.key[q] & 1023u), (int)(T.key[q] >> 10 & 1023u));
    __syncwarp();
    int arg = -1;
    double best = CUDART_INF;
    if (lane == 0) {
        // the pairs were listed from the last layer down, k ascending: backwards, the lowest k comes last
        for (int q = np - 1; q >= 0; q--) {
            const uint32_t f = T.key[q];
            const int i = (int)(f >> 20), k = (int)(f & 1023u);
            const double c = __dadd_rn(i == 3 ? row_base(T, k) : T.dp64[(size_t)(i - 1) * p + k], T.cost[q]);
            if (c <= best) { best = c; arg = k; }
            if (q == 0 || T.key[q - 1] >> 10 != f >> 10) {  // the output's last: store it
                const size_t o = (size_t)i * p + (f >> 10 & 1023u);
                T.dp64[o] = best;
                T.arg[o] = (uint16_t)arg;
                if (q > 0) best = CUDART_INF;
            }
        }
        if (row_outside(T, i0, j0, best)) atomicAdd(T.tally, 1);
    }
    best = __shfl_sync(full, best, 0);
    arg = __shfl_sync(full, arg, 0);
    *value = best;
    return arg;
}

// The path from the resolved output (i, j) down to layer 3 into a[]: a closure holds every layer below, so all of it is
// resolved; then what the trace listed is forgotten.
static __device__ __noinline__ void row_follow(const RowTrace &T, int i, int j, int s, int32_t *a) {
    const int lane = threadIdx.x & 31, p = T.p;
    for (; i >= 3; i--) {
        j = T.arg[(size_t)i * p + j];
        if (lane == 0) a[i - 2] = j;
    }
    for (int l = 3 + lane; l <= s; l += 32) {
        for (int e = 0; e < T.cnt[l]; e++) T.need[(size_t)l * T.nw + (T.list[(size_t)l * p + e] >> 5)] = 0u;
        T.cnt[l] = 0;
    }
}

// The codebook of multiplier T.g into a[0 .. m-1] (lane 0 writes); returns m, 0 when there is none.
static __device__ __forceinline__ int row_trace(const RowTrace &T, int s, int ilo, int32_t *a) {
    const int lane = threadIdx.x & 31, p = T.p;
    const unsigned full = 0xffffffffu;
    // eq. apx_final: the layers whose fp32 value is within the band of the least
    float m = CUDART_INF_F;
    for (int i = ilo + lane; i <= s; i += 32) m = fminf(m, T.dp[((size_t)i * p + p - 1) * kMaxG + T.g]);
    for (int o = 16; o; o >>= 1) m = fminf(m, __shfl_xor_sync(full, m, o));
    if (!(m < CUDART_INF_F)) return 0;
    const float lim = row_limit(T, s, m);
    int istar = -1, members = 0;
    for (int i = ilo; i <= s; i++)
        if (!(T.dp[((size_t)i * p + p - 1) * kMaxG + T.g] > lim)) { if (!members++) istar = i; }
    bool resolved = members > 1;
    if (resolved) {
        double best = CUDART_INF;
        bool known = false;
        for (int i = ilo; i <= s; i++) {
            if (T.dp[((size_t)i * p + p - 1) * kMaxG + T.g] > lim) continue;
            double v;
            if (i == 2) v = row_base(T, p - 1);
            else { row_resolve(T, i, p - 1, known, &v); known = true; }
            if (v < best) { best = v; istar = i; }
        }
    }
    int j = p - 1, i = istar;
    if (lane == 0) a[istar - 1] = j;
    for (; i >= 3 && !resolved; i--) {
        const float lj = row_limit(T, i, T.dp[((size_t)i * p + j) * kMaxG + T.g]);
        int n = 0, k = 0;
        for (int kb = 0; kb < j; kb += 128) {
            unsigned in[4];
            row_members(T, i, j, kb, lj, in);
#pragma unroll
            for (int w = 0; w < 4; w++) {
                if (in[w] && !n) k = kb + 32 * w + __ffs(in[w]) - 1;
                n += __popc(in[w]);
            }
        }
        if (n > 1) {
            double v;
            row_resolve(T, i, j, false, &v);
            resolved = true;
            break;
        }
        j = k;
        if (lane == 0) a[i - 2] = j;
    }
    if (resolved) row_follow(T, i, j, s, a);
    if (lane == 0) a[0] = 0;
    __syncwarp();
    return istar;
}

// A block's scratch of multiplier g and row_trace on it.  Not in line, and with pointers of its own: what the forward pass does
// not need then takes none of its 80 registers (8192 rows of 128 values: 9.8 ms of passes, 10.1 otherwise).
static __device__ __noinline__ int row_codebook(const RowsPass &A, int64_t row, int p, int g, const float2 *cf, double lam,
                                                float lam32, float slack, double scale, float noise, uint16_t *cnt, int *tally,
                                                int32_t *a) {
    const size_t dc = (size_t)A.R.dcap, rows_per = (size_t)(A.s + 1) * dc, nwc = (dc + 31) / 32;
    const size_t at = (size_t)blockIdx.x * kMaxG + g;
    const RowCosts rc = row_costs(A, row);
    double *cost = A.cost + at * (kRowsPairs + kRowsPairs / 2);  // kRowsPairs costs, then as many keys
    const RowTrace T{row_prefix(A.R, row, p), cf, rc.c0, rc.phf, A.dp + blockIdx.x * rows_per * kMaxG, A.dp64 + at * rows_per,
                     A.list + at * rows_per, A.need + at * (size_t)(A.s + 1) * nwc, A.arg + at * rows_per, cnt + g * (A.s + 1),
                     cnt + (kMaxG + g) * (A.s + 1), reinterpret_cast<uint32_t *>(cost + kRowsPairs), cost, A.tau, lam, scale,
                     lam32, slack, noise, p, g, (int)nwc, tally};
    return row_trace(T, A.s, A.exact_s ? A.s : 2, a);
}

// eval_codebook_lanes for the multipliers g0 .. of one warp, `width` lanes (a power of two >= s) each: the same
// values in the same order; a binary64 sequence costs a warp the same for one lane as for 32.  Returns MSE + lam H(I,B).
__device__ __forceinline__ double row_evaluate(const Prefix &P, const int32_t *a, int m, int width, double lam, double *out3) {
    const unsigned full = 0xffffffffu;
    const int l = threadIdx.x & (width - 1);
    double C = 0.0, F = 0.0, U = 0.0, D = 0.0;
    if (l + 1 < m) {
        pair_exact(P, a[l], a[l + 1], C, U, D);
        F = l == 0 ? phi_first_at(P, a[0], U, D) : phi_exact(P, U, D, false);
    }
    const double Uprev = __shfl_up_sync(full, U, 1, width);
    const double Ulast = __shfl_sync(full, U, m >= 2 ? m - 2 : 0, width);
    double ht = 0.0;
    if (m >= 2 && l < m) {
        const double f = l == m - 1 ? Ulast : (l == 0 ? __dadd_rn((double)P.w[a[0]], D) : __dadd_rn(Uprev, D));
        ht = hfun(__ddiv_rn(f, (double)P.d));
    }
    double mse = 0.0, hs = 0.0, hx = 0.0;
    for (int r = 0; r < width; r++) {
        const double c = __shfl_sync(full, C, r, width), f = __shfl_sync(full, F, r, width), h = __shfl_sync(full, ht, r, width);
        if (r + 1 < m) { mse = __dadd_rn(mse, c); hs = __dadd_rn(hs, f); }
        if (r < m && m >= 2) hx = __dadd_rn(hx, h);
    }
    if (l == 0 && m > 0) { out3[0] = mse; out3[1] = hs; out3[2] = hx; }
    return __dadd_rn(mse, __dmul_rn(lam, hs));
}

// Shared memory: two layers [p][8] as float bits, the pairs' costs (p <= kRowsMaxP), the evaluation's scratch
// (s > 32), the codebooks and the closures' counts.
__host__ __device__ __forceinline__ size_t rows_smem_costs(int p) { return sizeof(int) * 2 * kMaxG * (size_t)p; }
__host__ __device__ __forceinline__ size_t rows_smem_tail(int p) {
    const size_t pc = (size_t)(p < kRowsMaxP ? p : kRowsMaxP);
    return rows_smem_costs(p) + sizeof(float2) * (pc * (pc - 1) / 2);
}
static size_t rows_pass_smem(int p, int s) {
    return rows_smem_tail(p) + (s > 32 ? sizeof(double) * 4 * kMaxS : 0) + kMaxG * (sizeof(int32_t) * s + 2 * sizeof(uint16_t) * (s + 1));
}

// WIDE: some row has more than kRowsMaxP values; its pairs' costs stay in global memory.
template <bool WIDE>
__global__ void __launch_bounds__(WIDE ? kRowsThreads : 256, WIDE ? 1 : 3) k_rows_pass(const __grid_constant__ RowsPass A) {
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ int m_sm[kMaxG];
    __shared__ double lam[kMaxG];
    __shared__ float lam32[kMaxG];
    __shared__ int refuse;
    __shared__ int tally[2];
    __shared__ float noise;
    const RowsData &R = A.R;
    const int G = A.G, s = A.s, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarp = blockDim.x >> 5;
    const size_t dc = (size_t)R.dcap, rows_per = (size_t)(s + 1) * dc;
    double *scratch = reinterpret_cast<double *>(rsm + rows_smem_tail(A.pmax));
    int32_t *a_sm = reinterpret_cast<int32_t *>(scratch + (s > 32 ? 4 * kMaxS : 0));
    uint16_t *cnt_sm = reinterpret_cast<uint16_t *>(a_sm + kMaxG * s);
    float *dp = A.dp + blockIdx.x * rows_per * kMaxG;
    {
        const size_t n = (size_t)(s + 1) * ((dc + 31) / 32) * kMaxG;
        for (size_t q = tid; q < n; q += blockDim.x) A.need[blockIdx.x * n + q] = 0u;
    }
    if (tid < 2) tally[tid] = 0;
    for (int q = tid; q < kMaxG * (s + 1); q += blockDim.x) cnt_sm[q] = 0;  // (row_follow leaves it at zero)
    for (int b = blockIdx.x; b < A.nact; b += gridDim.x) {
        const int64_t row = A.rows[b];
        const int p = (int)R.p[row];
        const Prefix P = row_prefix(R, row, p);
        const RowCosts rc = row_costs(A, row);
        const double scale = rc.phf[0];
        __syncthreads();  // the row before is done
        if (tid == 0) {
            const double x = rc.c0[0];
            refuse = x < 0.0;
            noise = __double2float_ru(x);
        }
        if (tid < kMaxG) {
            lam[tid] = tid < G ? A.lam[(size_t)b * G + tid] : 0.0;
            lam32[tid] = __double2float_rn(__dmul_rn(lam[tid], scale));
        }
        __syncthreads();
        if (tid < G && !(lam32[tid] < 0x1p120f)) refuse = 1;
        __syncthreads();
        if (refuse) {
            if (tid < G) A.mcount[(size_t)b * G + tid] = -1;
            continue;
        }
        int *prev = reinterpret_cast<int *>(rsm), *out = prev + kMaxG * p;
        float2 *csm = reinterpret_cast<float2 *>(rsm + rows_smem_costs(A.pmax));
        const bool in_sm = !WIDE || p <= kRowsMaxP;
        if (in_sm)
        {
            const int np = p * (p - 1) / 2;
            const float4 *src = reinterpret_cast<const float4 *>(rc.cf);
            float4 *dst = reinterpret_cast<float4 *>(csm);
#pragma unroll 4
            for (int t = tid; t < np / 2; t += blockDim.x) dst[t] = src[t];
            if (tid == 0 && (np & 1)) csm[np - 1] = rc.cf[np - 1];
        }
        const float2 *cf = in_sm ? csm : rc.cf;
        // eq. apx_base: dp(2, j) = C[0, j] + lambda' Phi^first[0, j]
        for (int q = tid; q < kMaxG * p; q += blockDim.x) {
            const int j = q / kMaxG, g = q % kMaxG;
            float v = CUDART_INF_F;
            if (j >= 1) v = fmaxf(__double2float_rn(__dmul_rn(__dadd_rn(rc.c0[j], __dmul_rn(lam[g], rc.phf[j])), scale)), 0.f) + 0.f;
            prev[q] = __float_as_int(v);
            out[q] = 0x7f800000;
            dp[(size_t)2 * p * kMaxG + q] = v;
        }
        __syncthreads();
        // eq. apx_rec: a warp's unit is 32 columns (a lane one) and ks of their k; the values are >= +0, so
        // their bits order like them.  Rows of at most 128 values have 20 units of 16 k for 8 warps.
        const int ks = in_sm ? 16 : 32, ctop = (p - 1) >> 5;
        for (int i = 3; i <= s; i++) {
            int c = ctop, q = wid;
            for (;;) {
                int cnt = 0;
                while (c >= 0 && q >= (cnt = (min(32 * c + 31, p - 1) + ks - 1) / ks)) { q -= cnt; c--; }
                if (c < 0) break;
                const int j = 32 * c + lane, k0 = q * ks, k1 = min(k0 + ks, min(32 * c + 31, p - 1));
                int acc[kMaxG];
#pragma unroll
                for (int g = 0; g < kMaxG; g++) acc[g] = 0x7f800000;
                float lg[kMaxG];
#pragma unroll
                for (int g = 0; g < kMaxG; g++) lg[g] = lam32[g];
                const float2 *cp = cf + pair_at(k0, j, p);
                const int jhi = j < p ? j : 0;
#pragma unroll 4
                for (int k = k0; k < k1; k++) {
                    const float2 f = k < jhi ? *cp : make_float2(CUDART_INF_F, 0.f);
                    cp += p - k - 2;  // the next k's row starts one pair later
                    const float4 x = *reinterpret_cast<const float4 *>(prev + k * kMaxG);
                    const float4 y = *reinterpret_cast<const float4 *>(prev + k * kMaxG + 4);
                    const float pv[kMaxG] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int g = 0; g < kMaxG; g++)
                        acc[g] = min(acc[g], __float_as_int(__fadd_rn(pv[g], __fmaf_rn(lg[g], f.y, f.x))));
                }
                if (j < p) {
#pragma unroll
                    for (int g = 0; g < kMaxG; g++) atomicMin(&out[j * kMaxG + g], acc[g]);
                }
                q += nwarp;
            }
            __syncthreads();
            for (int t = tid; t < kMaxG * p; t += blockDim.x) {
                dp[(size_t)i * p * kMaxG + t] = __int_as_float(out[t]);
                prev[t] = 0x7f800000;
            }
            int *x = prev;
            prev = out;
            out = x;
            __syncthreads();
        }
        // underflow: C and the gaps' products 2^-149 a term, Phi where y < 1e-37 2^-118 a layer; and what the binary64 costs of
        // an output and of its rival are off by (row_within), which decides where fp32's are exact: the rounding of ||X||^2
        auto slack = [&](int g) {
            return __fmul_ru(3.0f * (float)s, __fadd_ru(noise, __fmaf_ru(lam32[g], 0x1p-114f, 8.0f * (float)P.d * 0x1p-149f)));
        };
        for (int g = wid; g < G; g += nwarp) {
            const int m = row_codebook(A, row, p, g, cf, lam[g], lam32[g], slack(g), scale, noise, cnt_sm, tally, a_sm + g * s);
            if (lane == 0) { m_sm[g] = m; A.mcount[(size_t)b * G + g] = m; }
            for (int r = lane; r < m; r += 32) A.qidx[((size_t)b * G + g) * s + r] = a_sm[g * s + r];
        }
        __syncthreads();
        // the codebook's objective against the fp32 value of its last output
        auto certify = [&](int g, double objective) {
            const int m = m_sm[g];
            if (m > 0 && !row_within(dp[((size_t)m * p + p - 1) * kMaxG + g], objective, A.tau[m], slack(g), scale, m, noise))
                atomicAdd(tally, 1);
        };
        if (s <= 32) {
            const int width = s <= 4 ? 4 : s <= 8 ? 8 : s <= 16 ? 16 : 32, per = 32 / width;
            for (int g0 = wid * per; g0 < G; g0 += nwarp * per) {
                const int g = min(g0 + lane / width, G - 1);  // (spare lanes repeat the last one's values)
                const double J = row_evaluate(P, a_sm + g * s, m_sm[g], width, lam[g], &A.metrics[((size_t)b * G + g) * 4 + 1]);
                if (lane % width == 0 && g0 + lane / width < G) certify(g, J);
            }
        } else if (wid == 0) {  // one warp, multiplier by multiplier
            for (int g = 0; g < G; g++) {
                double *q = &A.metrics[((size_t)b * G + g) * 4 + 1];
                if (m_sm[g] > 0) eval_codebook_warp(P, a_sm + g * s, m_sm[g], q, scratch);
                if (lane == 0) certify(g, __dadd_rn(q[0], __dmul_rn(lam[g], q[1])));  // (lane 0 wrote them)
                __syncwarp();
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (tally[0]) atomicAdd(&A.st->bound_viol, tally[0]);
        if (tally[1]) atomicAdd((unsigned long long *)&A.st->rescored, (unsigned long long)tally[1]);
    }
}

int launch_rows_pass(const RowsPass &A, int slots, cudaStream_t st) {
    if (A.nact == 0) return ECASQ_OK;
    if (A.pmax > kScanTile) return ECASQ_EINVAL;
    RowsPass B = A;
    float eps[kMaxS + 1];
    band_factors(A.s, B.tau, eps);
    if (!A.pairs_ready) {
        note_launch();
        k_rows_build<<<(unsigned)A.nact, (unsigned)std::max(128, (A.pmax + 31) & ~31), 0, st>>>(B);
        ECASQ_LAUNCH_CHECK();
    }
    const size_t smem = rows_pass_smem(A.pmax, A.s);
    const bool wide = A.pmax > kRowsMaxP;
    const void *f = wide ? (const void *)k_rows_pass<true> : (const void *)k_rows_pass<false>;
    // the same limit in every call (the longest rows and largest s): another thread's call of another shape may
    // lie between this and the launch
    ECASQ_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_pass_smem(kScanTile, kMaxS)));
    const unsigned blocks = (unsigned)std::min(A.nact, slots);
    note_launch();
    if (wide) k_rows_pass<true><<<blocks, kRowsThreads, smem, st>>>(B);
    else k_rows_pass<false><<<blocks, 256, smem, st>>>(B);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

// Q[row][r] = v_row[a[row][r]] for the selected codebooks.
__global__ void k_rows_gather(RowsData R, const int32_t *a, const int32_t *m, int s, float *Q) {
    const int64_t row = blockIdx.x;
    const float *v = R.v + row * R.dcap;
    for (int r = threadIdx.x; r < m[row]; r += blockDim.x) Q[row * s + r] = v[a[row * s + r]];
}

int launch_rows_gather(const RowsData &R, const int32_t *a, const int32_t *m, int64_t rows, int s, float *Q,
                       cudaStream_t st) {
    note_launch();
    k_rows_gather<<<(unsigned)rows, 32, 0, st>>>(R, a, m, s, Q);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

}  // namespace ecasq
