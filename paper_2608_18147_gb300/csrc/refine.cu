// refine.cu -- one colour step of the three-colour refinement (Sec. 6).
//
// Block b moves the b-th value of the colour class: q_l with l % 3 == colour,
// 1 <= l <= m-2.  Its candidates are the unique input values strictly between
// its fixed neighbours; the local objective of Sec. 6 (true entropy reading) is
//   C[q_{l-1}, c] + C[c, q_{l+1}] + lambda' (h(f_{l-1}/d) + h(f_l/d) + h(f_{l+1}/d)),
// f_{l-1} = U[q_{l-2}, q_{l-1}] + D[q_{l-1}, c]   (n_{q_0} + D[q_0, c] when l-1 = 0),
// f_l     = U[q_{l-1}, c] + D[c, q_{l+1}],
// f_{l+1} = U[c, q_{l+1}] + D[q_{l+1}, q_{l+2}]   (U[c, q_{m-1}] when l+1 = m-1).
// Values of one class never share a frequency term, so all of them move at
// once (Sec. 6, Fig. 3).  Ties keep the current value, else the lowest index.
//
// The scan of q_l is a function of (q_{l-2}, q_{l-1}, q_l, q_{l+1}, q_{l+2}) alone (and of
// lambda', fixed in a call).  ctx[l] records that context whenever a scan kept q_l
// where it was; while the context is unchanged the scan would keep it again, so the
// value is not scanned (same result, no candidate evaluated).  A value that moved has
// no record (its move may still be undone by the caller).
#include "common.cuh"
#include "cost32.cuh"

namespace ecasq {

constexpr int kCtx = 6;  // q_{l-2}, q_{l-1}, q_l, q_{l+1}, q_{l+2} (-1 past the ends), valid

__device__ __forceinline__ void context_of(const int32_t *a, int m, int l, int32_t c[5]) {
    c[0] = l >= 2 ? a[l - 2] : -1;
    c[1] = a[l - 1];
    c[2] = a[l];
    c[3] = a[l + 1];
    c[4] = l + 2 <= m - 1 ? a[l + 2] : -1;
}
__device__ __forceinline__ bool context_unchanged(const int32_t *a, int m, int l, const int32_t *ctx) {
    const int32_t *r = ctx + kCtx * l;
    if (!r[5]) return false;
    int32_t c[5];
    context_of(a, m, l, c);
    return c[0] == r[0] && c[1] == r[1] && c[2] == r[2] && c[3] == r[3] && c[4] == r[4];
}

struct Nbr {
    int64_t L, R, cur, a0;
    double Ux, Dx;   // outer neighbours' fixed halves of f_{l-1} and f_{l+1}
    int firstL, lastR;
};

__device__ __forceinline__ double local_obj(const Prefix &P, const Nbr &n, int64_t c, double lamp) {
    double dd_ = (double)P.d;
    double C1, U1, D1, C2, U2, D2;
    pair_exact(P, n.L, c, C1, U1, D1);
    pair_exact(P, c, n.R, C2, U2, D2);
    double fl = n.firstL ? __dadd_rn((double)P.w[n.a0], D1) : __dadd_rn(n.Ux, D1);
    double fm = __dadd_rn(U1, D2);
    double fr = n.lastR ? U2 : __dadd_rn(U2, n.Dx);
    double ent = __dadd_rn(__dadd_rn(hfun(__ddiv_rn(fl, dd_)), hfun(__ddiv_rn(fm, dd_))), hfun(__ddiv_rn(fr, dd_)));
    return __dadd_rn(__dadd_rn(C1, C2), __dmul_rn(lamp, ent));
}

constexpr int kRefineChunk = 256;   // candidates per block, at most, one per thread (chunk_of)

struct RefPart { double v; int64_t i; };
constexpr int kRefineValues = kMaxS / 3 + 1;  // values of one colour class, at most

// A value's scan: its neighbours, an upper bound of its least objective and the error bounds of the screening.
struct RefineScan {
    Nbr n;
    double ub;           // the least exact objective of some candidates, the current position among them
    double vL, vR, S, S2, nT, T, T2, scale;  // v, S, S2 of the neighbours' interval; 2^-e for fp32
    int64_t N;
    float lam, errC, errU, invd, wfirst, Ux, Dx;
};

// The neighbours of value l (whole warp: the two outer intervals side by side).
__device__ __forceinline__ Nbr make_nbr(const Prefix &P, const int32_t *a, int m, int l) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    Nbr n;
    n.L = a[l - 1]; n.R = a[l + 1]; n.cur = a[l]; n.a0 = a[0];
    n.firstL = (l - 1 == 0); n.lastR = (l + 1 == m - 1);
    double C, U = 0.0, D = 0.0;
    if (lane == 0 && !n.firstL) pair_exact(P, a[l - 2], n.L, C, U, D);
    if (lane == 1 && !n.lastR) pair_exact(P, n.R, a[l + 2], C, U, D);
    n.Ux = __shfl_sync(full, U, 0);
    n.Dx = __shfl_sync(full, D, 1);
    if (n.firstL) n.Ux = 0.0;
    if (n.lastR) n.Dx = 0.0;
    return n;
}

// One warp per value: the exact objective at the current position (curval) and at 31 others, around it and
// across the range, as a binary64 sequence costs a warp the same for one lane as for 32.
__global__ void __launch_bounds__(32) k_refine_bound(Prefix P, const int32_t *a, int m, int colour, double lamp,
                                                     double *curval, RefineScan *scan, const int32_t *ctx) {
    const int lane = threadIdx.x, l = (colour == 0 ? 3 : colour) + 3 * blockIdx.x;
    if (l > m - 2 || context_unchanged(a, m, l, ctx)) return;
    const unsigned full = 0xffffffffu;
    const Nbr n = make_nbr(P, a, m, l);
    int64_t c = n.cur;
    if (lane >= 16) c = n.L + 1 + (n.R - n.L - 1) * (2 * (lane - 16) + 1) / 32;
    else if (lane) c += (lane & 1 ? 1 : -1) * ((int64_t)1 << (lane - 1));
    c = min(max(c, n.L + 1), n.R - 1);
    const double v = local_obj(P, n, c, lamp);
    if (lane == 0) curval[blockIdx.x] = v;
    double ub = v;
    for (int o = 16; o; o >>= 1) ub = fmin(ub, __shfl_xor_sync(full, ub, o));
    if (lane == 0) {
        RefineScan q;
        q.n = n;
        q.ub = ub;
        q.vL = (double)P.v[n.L];
        q.vR = (double)P.v[n.R];
        q.N = P.N[n.L + 1];
        q.nT = (double)(P.N[n.R + 1] - q.N);
        const dd s0 = load_dd(P.S, P.p, n.L + 1), s1 = load_dd(P.S, P.p, n.R + 1);
        const dd q0 = load_dd(P.S2, P.p, n.L + 1), q1 = load_dd(P.S2, P.p, n.R + 1);
        q.T = (s1.hi - s0.hi) + (s1.lo - s0.lo);
        q.T2 = (q1.hi - q0.hi) + (q1.lo - q0.lo);
        // the screening's errors (k_refine_chunks), u = 2^-53, with V the larger magnitude of the two neighbours
        const double u = 0x1p-53, V = fmax(fabs(q.vL), fabs(q.vR)), NV = q.nT * V, NV2 = NV * V, d = (double)P.d;
        const double eS = 8 * u * (NV + 2 * u * (fabs(s0.hi) + fabs(s1.hi) + NV)), eQ = 8 * u * (NV2 + 2 * u * q1.hi);
        const double big = fmax(NV2, lamp);
        q.scale = big > 0.0 && isfinite(big) ? ldexp(1.0, -ilogb(big)) : 1.0;
        q.lam = __double2float_ru(lamp * q.scale);
        q.errC = __double2float_ru((16 * (V * eS + eQ + u * NV2) + 0x1p-45 * (NV2 + lamp)) * q.scale * 1.01);
        q.errU = __double2float_ru(124 * (3 * eS + 4 * u * NV) / d * 1.01);
        q.invd = 1.0f / (float)P.d;
        q.wfirst = n.firstL ? (float)P.w[n.a0] : 0.f;
        q.Ux = (float)n.Ux;
        q.Dx = (float)n.Dx;
        scan[blockIdx.x] = q;
    }
}

// Block (chunk, b): the b-th value of the colour class, candidates
// L+1+chunk*kRefineChunk .. (excluding the current position); the best
// (value, lowest index) of the chunk goes to part[b * nchunk + chunk].
//
// Only a candidate whose objective may be at or below the value's upper bound is evaluated as the
// definition asks, in double-double; the screening takes plain binary64 differences of the prefix sums for the
// costs and fp32 for the frequencies and their entropies.  Its error, over all candidates of the value
// (N entries between the neighbours, V the larger magnitude of the two, u = 2^-53):
//  * a difference of S is within eS = 8u (N V + 2u |S|), of S2 within eQ = 8u (N V^2 + 2u S2): the high words' difference
//    errs relative to itself, the low words are u of the sums;
//  * C = v_j A - (dS2 - v_k dS), A = dS - v_k n: two of them within 16 (V eS + eQ + u N V^2) (errC, which also holds
//    2^-45 of the objective's size for the evaluation's own roundings);
//  * a frequency f = U + D errs by at most 2 (3 eS + 4u N V) / (least distance to a neighbour) from its numerators, and
//    h(f/d) by 62 times that over d (h's slope where the argument is above 2^-60; below, h itself is
//    less than 2^-50) (errU);
//  * fp32: a quotient, a sum and a product leave f/d within 6 2^-24 of itself, h = -y log2 y thereby within
//    1.45 times that, __log2f errs by 2^-22 for y in [1/2, 2] and 2 ulp below, so three of them are within 2^-18, and the
//    products with lambda' and the sums within 2^-22 of their terms.
// What bounded it: 87 000 candidates a step at p = 131072, m = 16 at some 800 binary64 instructions each (2 a
// cycle and SM): 105 us; about one in a hundred is left to evaluate, and bound and scan take 51.  Without
// the screening (SCREEN false) every candidate is evaluated and the current position's goes to curval: 22 us at
// p = 1024 with blocks of 32 (38 with 256: eight sequences on one SM), against 42 for bound and scan.
template <int CHUNK, bool SCREEN>
__global__ void __launch_bounds__(CHUNK) k_refine_chunks(Prefix P, const int32_t *a, int m, int colour, double lamp,
                                                                const RefineScan *scan, double *curval, RefPart *part,
                                                                int nchunk, const int32_t *ctx) {
    __shared__ int list[CHUNK];
    __shared__ Nbr nb;
    __shared__ int count;
    __shared__ double rv[CHUNK / 32];
    __shared__ int64_t ri[CHUNK / 32];
    const int l = (colour == 0 ? 3 : colour) + 3 * blockIdx.y;
    if (l > m - 2) return;
    const int64_t lo = (int64_t)a[l - 1] + 1 + (int64_t)blockIdx.x * CHUNK;
    const int64_t hi = min((int64_t)a[l + 1], lo + CHUNK);
    if (lo >= hi || context_unchanged(a, m, l, ctx)) return;  // uniform over the block
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const RefineScan &q = scan[blockIdx.y];
    const int64_t c = lo + threadIdx.x;
    if (wid == 0) {
        const Nbr x = SCREEN ? q.n : make_nbr(P, a, m, l);
        if (lane == 0) { nb = x; count = 0; }
    }
    __syncthreads();
    bool in = false;
    if (SCREEN && c < hi && c != q.n.cur) {
        const double vc = (double)P.v[c], n1 = (double)(P.N[c + 1] - q.N), n2 = q.nT - n1;
        const dd s = load_dd(P.S, P.p, c + 1), s2 = load_dd(P.S2, P.p, c + 1);
        const dd s0 = load_dd(P.S, P.p, q.n.L + 1), q0 = load_dd(P.S2, P.p, q.n.L + 1);
        const double dS = (s.hi - s0.hi) + (s.lo - s0.lo), dQ = (s2.hi - q0.hi) + (s2.lo - q0.lo);
        const double eS = q.T - dS, eQ = q.T2 - dQ;
        const double A1 = __fma_rn(-q.vL, n1, dS), E1 = __fma_rn(vc, n1, -dS), C1 = __fma_rn(vc, A1, __fma_rn(q.vL, dS, -dQ));
        const double A2 = __fma_rn(-vc, n2, eS), E2 = __fma_rn(q.vR, n2, -eS), C2 = __fma_rn(q.vR, A2, __fma_rn(vc, eS, -eQ));
        const float x = (float)((C1 + C2 - q.ub) * q.scale);
        const float r1 = 1.0f / __double2float_rd(vc - q.vL), r2 = 1.0f / __double2float_rd(q.vR - vc);
        const float U1 = fmaxf((float)A1, 0.f) * r1, D1 = fmaxf((float)E1, 0.f) * r1;
        const float U2 = fmaxf((float)A2, 0.f) * r2, D2 = fmaxf((float)E2, 0.f) * r2;
        const float yl = (q.n.firstL ? q.wfirst + D1 : q.Ux + D1) * q.invd, ym = (U1 + D2) * q.invd;
        const float yr = (q.n.lastR ? U2 : U2 + q.Dx) * q.invd;
        const float ent = yl * -__log2f(fmaxf(yl, 1e-37f)) + ym * -__log2f(fmaxf(ym, 1e-37f)) + yr * -__log2f(fmaxf(yr, 1e-37f));
        const float err = q.errC + q.lam * (0x1p-18f + fabsf(ent) * 0x1p-22f + q.errU * (r1 + r2)) * 1.01f + fabsf(x) * 0x1p-22f;
        in = !(x + q.lam * ent > err);  // (a value out of the fp32 range stays in)
    }
    if (SCREEN) {
        const unsigned b = __ballot_sync(0xffffffffu, in);
        int at = 0;
        if (lane == 0 && b) at = atomicAdd(&count, __popc(b));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) list[at + __popc(b & ((1u << lane) - 1u))] = threadIdx.x;
        __syncthreads();
    }
    const int n = SCREEN ? count : (int)(hi - lo);
    double bv = CUDART_INF;
    int64_t bi = -1;
    if ((int)threadIdx.x < n) {
        bi = SCREEN ? lo + list[threadIdx.x] : c;
        bv = local_obj(P, nb, bi, lamp);
        if (!SCREEN && bi == nb.cur) {
            curval[blockIdx.y] = bv;
            bv = CUDART_INF;
        }
        if (!(bv < CUDART_INF)) bi = -1;
    }
    if (32 * wid < n) {
        const int64_t own = bi;
        long long key = order_key(bv);  // of +inf where there is no candidate
        int64_t i = bi < 0 ? INT64_MAX : bi;
        for (int o = 16; o > 0; o >>= 1) {
            const long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
            const int64_t i2 = __shfl_xor_sync(0xffffffffu, i, o);
            if (k2 < key || (k2 == key && i2 < i)) { key = k2; i = i2; }
        }
        const unsigned has = __ballot_sync(0xffffffffu, own == i);
        bv = __shfl_sync(0xffffffffu, bv, has ? __ffs(has) - 1 : 0);
        bi = has ? i : -1;
    }
    if (lane == 0) { rv[wid] = bv; ri[wid] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; 32 * w < n; w++)
            if (ri[w] >= 0 && (bi < 0 || rv[w] < bv || (rv[w] == bv && ri[w] < bi))) { bv = rv[w]; bi = ri[w]; }
        part[(size_t)blockIdx.y * nchunk + blockIdx.x] = {bv, bi};
    }
}

// One block per moved value: best over the chunks (lowest index among equal
// values), then keep the current position unless the best is strictly lower.
constexpr int kPickThreads = 256;
__global__ void __launch_bounds__(kPickThreads) k_refine_pick(const int32_t *a, int m, int colour, const RefPart *part, const double *curval,
                              int nchunk, int chunk, int32_t *a_new, int32_t *moved, int32_t *ctx) {
    int l0 = colour == 0 ? 3 : colour;
    int l = l0 + 3 * blockIdx.x;
    if (l > m - 2) return;
    if (context_unchanged(a, m, l, ctx)) return;  // a_new[l] == a[l] already
    int64_t range = (int64_t)a[l + 1] - (int64_t)a[l - 1] - 1;
    int nc = (int)cdiv(range, chunk);
    __shared__ double rv[kPickThreads / 32];
    __shared__ int64_t ri[kPickThreads / 32];
    double bv = CUDART_INF;
    int64_t bi = INT64_MAX;
    auto meet = [&](double v2, int64_t i2) {  // binary64 compares as integers (order_key)
        const long long k2 = order_key(v2), k = order_key(bv);
        if (i2 >= 0 && (k2 < k || (k2 == k && i2 < bi))) { bv = v2; bi = i2; }
    };
    for (int c = threadIdx.x; c < nc; c += kPickThreads) {
        const RefPart q = part[(size_t)blockIdx.x * nchunk + c];
        meet(q.v, q.i);
    }
    for (int o = 16; o > 0; o >>= 1) meet(__shfl_xor_sync(0xffffffffu, bv, o), __shfl_xor_sync(0xffffffffu, bi, o));
    if ((threadIdx.x & 31) == 0) { rv[threadIdx.x >> 5] = bv; ri[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kPickThreads / 32; w++) meet(rv[w], ri[w]);
        if (bi == INT64_MAX) bi = -1;
    }
    if (threadIdx.x == 0) {
        const int64_t cur = a[l];
        const double vc = curval[blockIdx.x];  // local_obj at the current position (k_refine_bound)
        int64_t nw = (bi >= 0 && bv < vc) ? bi : cur;
        a_new[l] = (int32_t)nw;
        if (nw != cur) atomicExch(moved, 1);
        int32_t *r = ctx + kCtx * l;
        if (nw == cur) {
            int32_t c[5];
            context_of(a, m, l, c);
            for (int q = 0; q < 5; q++) r[q] = c[q];
            r[5] = 1;
        } else {
            r[5] = 0;
        }
    }
}

// After a colour step: the step's codebook replaces the current one unless no value moved,
// or (with the guard) its H(Xhat), ev[2] from the gated evaluation, exceeds the budget
// (Sec. 6).  On the device, so that a refinement round needs no host round trip until
// its stop test.
// A value that moved went to the lowest-index minimiser of its local objective, which does
// not depend on the value itself, only on its four neighbours (other colours: they did not
// move in this step); a scan in its new context would keep it there, so a kept step gives
// it the record such a scan writes, and the next round does not scan it again unless a
// neighbour moves.
// kept: the evaluation of the current codebook, replaced with it, so that a round's stop test needs none of its own.
// a_new and moved are left as the next step starts: the current codebook, nothing moved.
__global__ void k_refine_commit(int32_t *a, int32_t *a_new, int32_t *moved, const double *ev, double *kept, int m,
                                int guard, double budget, int32_t *ctx) {
    if (*moved && !(guard && ev[2] > budget)) {
        for (int l = threadIdx.x; l < m; l += blockDim.x) {
            if (a_new[l] == a[l]) continue;
            int32_t c[5];
            context_of(a_new, m, l, c);
            int32_t *r = ctx + kCtx * l;
            for (int q = 0; q < 5; q++) r[q] = c[q];
            r[5] = 1;
        }
        __syncwarp();  // every comparison with the old codebook is done
        for (int t = threadIdx.x; t < m; t += blockDim.x) a[t] = a_new[t];
        if (threadIdx.x < 3) kept[threadIdx.x] = ev[threadIdx.x];
    } else {
        for (int t = threadIdx.x; t < m; t += blockDim.x) a_new[t] = a[t];
    }
    __syncwarp();
    if (threadIdx.x == 0) *moved = 0;
}

int launch_refine_commit(int32_t *a, int32_t *a_new, int32_t *moved, const double *ev, double *kept, int m, bool guard,
                         double budget, int32_t *ctx, cudaStream_t st) {
    note_launch();
    k_refine_commit<<<1, 32, 0, st>>>(a, a_new, moved, ev, kept, m, guard ? 1 : 0, budget, ctx);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

size_t refine_scratch_bytes(int64_t d) {
    return sizeof(double) * kRefineValues + sizeof(RefineScan) * kRefineValues +
           sizeof(RefPart) * kRefineValues * (size_t)cdiv(d, kRefineChunk);
}

size_t refine_ctx_bytes() { return sizeof(int32_t) * kCtx * kMaxS; }

int launch_refine_colour(const Prefix &P, const int32_t *a, int m, int colour, double lamp, int32_t *a_new,
                         int32_t *moved, void *part_buf, int32_t *ctx, int num_sms, cudaStream_t st, int *nblocks_out) {
    int l0 = colour == 0 ? 3 : colour;
    int nblk = (m - 2 >= l0) ? (m - 2 - l0) / 3 + 1 : 0;
    *nblocks_out = nblk;
    if (nblk == 0) return ECASQ_OK;
    // Screened above 512 candidates an SM, where the full scan's binary64 time passes bound and scan.  A
    // block's warps share an SM's binary64 pipe (a candidate's sequence is 5 us of it), so the blocks are as small as the
    // room for their results allows.
    const bool screen = P.p > (int64_t)512 * num_sms;
    int chunk = screen ? 64 : 32;
    while (chunk < kRefineChunk && nblk * cdiv(P.p, chunk) > kRefineValues * cdiv(P.d, kRefineChunk)) chunk *= 2;
    const int nchunk = (int)cdiv(P.p, chunk);
    double *curval = reinterpret_cast<double *>(part_buf);  // then the values' scans and the chunks' partial results
    RefineScan *scan = reinterpret_cast<RefineScan *>(curval + kRefineValues);
    RefPart *part = reinterpret_cast<RefPart *>(scan + kRefineValues);
    if (screen) {
        note_launch();
        k_refine_bound<<<nblk, 32, 0, st>>>(P, a, m, colour, lamp, curval, scan, ctx);
        ECASQ_LAUNCH_CHECK();
    }
    const dim3 grid(nchunk, nblk);
    note_launch();
    auto go = [&](auto kernel) { kernel<<<grid, chunk, 0, st>>>(P, a, m, colour, lamp, scan, curval, part, nchunk, ctx); };
    switch (chunk) {
        case 32: go(k_refine_chunks<32, false>); break;
        case 64: screen ? go(k_refine_chunks<64, true>) : go(k_refine_chunks<64, false>); break;
        case 128: screen ? go(k_refine_chunks<128, true>) : go(k_refine_chunks<128, false>); break;
        default: screen ? go(k_refine_chunks<256, true>) : go(k_refine_chunks<256, false>); break;
    }
    ECASQ_LAUNCH_CHECK();
    note_launch();
    k_refine_pick<<<nblk, kPickThreads, 0, st>>>(a, m, colour, part, curval, nchunk, chunk, a_new, moved, ctx);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

}  // namespace ecasq
