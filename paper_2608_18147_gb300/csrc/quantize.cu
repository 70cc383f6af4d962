// quantize.cu -- unbiased stochastic quantization (Sec. 2) and the index
// histogram behind the empirical entropy (Sec. 1).
//
// Entry i (original order) with a = max{q <= x}: if x == a it keeps a's index;
// otherwise it rounds up to the next value iff
//   fl32(fl32(k * 2^-24) * fl32(b - a)) < fl32(x - a),
// k = top 24 bits of SplitMix64(seed + (i+1) * 0x9E3779B97F4A7C15)
// (Steele, Lea and Flood 2014).  HBM-bound: 4 B read + 1 B written per entry;
// the codebook and the histogram live in shared memory.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace ecasq {

__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;

// Whether a codebook of m values is not strictly ascending (NaN included), over the block's threads.
__device__ __forceinline__ bool unsorted(const float *Q, int m) {
    bool b = false;
    for (int r = threadIdx.x + 1; r < m; r += blockDim.x) b |= !(Q[r] > Q[r - 1]);
    return b;
}

// The block's n counts are in o.acc.  With a ticket the last block hands them to o.counts, so that one copy
// to the host brings the status record and the counts behind it.
__device__ __forceinline__ void finish_counts(const QuantOut &o, int n) {
    __shared__ int last;
    if (!o.ticket) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(o.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int r = threadIdx.x; r < n; r += blockDim.x) o.counts[r] = __ldcg(o.acc + r);
}

// half: the largest power of two <= m - 1 (0 when m = 1); q[m .. 2 half - 1] hold NaN, which no
// entry passes (+inf would let +inf pass), so the search needs no bound test.  zc = seed +
// (i + 1) * gamma (mod 2^64) for entry i.
__device__ __forceinline__ int search_half(int m) { return m > 1 ? 1 << (31 - __clz(m - 1)) : 0; }

__device__ __forceinline__ int quant_one(float xv, uint64_t zc, const float *q, int m, int half, bool &bad) {
    if (!(xv >= q[0] && xv <= q[m - 1])) { bad = true; return 0; }
    int t = 0;  // largest t with q[t] <= x: one step per bit of m - 1, the same count in every lane
    for (int b = half; b; b >>= 1)
        if (q[t + b] <= xv) t += b;
    if (q[t] != xv) {
        uint64_t z = splitmix64(zc);
        float k = __fmul_rn((float)(uint32_t)(z >> 40), 0x1p-24f);
        float d1 = __fsub_rn(xv, q[t]);
        float d2 = __fsub_rn(q[t + 1], q[t]);
        if (__fmul_rn(k, d2) < d1) t += 1;
    }
    return t;
}

// Codebooks of at most kPrivBins values count their indices in per-thread
// histograms: 16-bit counters packed in pairs, word w of thread t at
// ph[w * 256 + t] (each thread its own bank column: no conflicts, no atomics).  A
// thread folds its counters into the block's 32-bit totals after every
// kFoldEntries of its entries, before any counter could pass 65535 (only inputs of
// more than about 10^10 entries get that far).
constexpr int kPrivBins = 32;
constexpr int kQThreads = 256;
constexpr int kFoldEntries = 32768;

__device__ __forceinline__ void priv_count(uint32_t *ph, int t) {
    ph[(t >> 1) * kQThreads + threadIdx.x] += 1u << ((t & 1) << 4);
}
__device__ __forceinline__ void priv_fold(uint32_t *ph, uint32_t *hcount, int m) {
    for (int w = 0; w < (m + 1) >> 1; w++) {
        const uint32_t v = ph[w * kQThreads + threadIdx.x];
        if (v) {
            if (v & 0xffffu) atomicAdd(&hcount[2 * w], v & 0xffffu);
            if (v >> 16) atomicAdd(&hcount[2 * w + 1], v >> 16);
            ph[w * kQThreads + threadIdx.x] = 0;
        }
    }
}

// Encode.  Vector path: each thread takes two groups of four entries per step (two
// 16-byte loads in flight before any arithmetic), writes four indices per group.
template <bool PRIV>
__global__ void __launch_bounds__(kQThreads) k_quantize(const float *__restrict__ x, int64_t d,
                                                        const float *__restrict__ Q, int m, uint64_t seed,
                                                        uint8_t *__restrict__ idx, QuantOut o) {
    __shared__ float q[kMaxS];
    __shared__ uint32_t hcount[kMaxS];
    __shared__ uint32_t ph[PRIV ? (kPrivBins / 2) * kQThreads : 1];
    for (int r = threadIdx.x; r < kMaxS; r += blockDim.x) {
        q[r] = r < m ? Q[r] : CUDART_NAN_F;
        hcount[r] = 0;
    }
    const int half = search_half(m);
    if (PRIV)
        for (int w = 0; w < kPrivBins / 2; w++) ph[w * kQThreads + threadIdx.x] = 0;
    if (__syncthreads_or(unsorted(Q, m))) {  // nothing is encoded
        if (threadIdx.x == 0) o.st->range_err = kUnsortedQ;
        d = 0;
    }
    auto count = [&](int t) {
        if (PRIV) priv_count(ph, t); else atomicAdd(&hcount[t], 1u);
    };
    bool bad = false;
    const bool vec = ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && ((reinterpret_cast<uintptr_t>(idx) & 3) == 0);
    const int64_t ngroups = vec ? d / 4 : 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    uchar4 *i4 = reinterpret_cast<uchar4 *>(idx);
    int since_fold = 0;  // entries counted since the last fold
    for (int64_t g = g0; g < ngroups; g += 2 * stride) {
        const int64_t h = g + stride;
        const bool two = h < ngroups;
        const float4 xa = x4[g];
        const float4 xb = two ? x4[h] : make_float4(0.f, 0.f, 0.f, 0.f);
        {
            const uint64_t z0 = seed + (uint64_t)(4 * g + 1) * kGamma;  // entries 4g .. 4g+3: z0 + r gamma
            const int t0 = quant_one(xa.x, z0, q, m, half, bad), t1 = quant_one(xa.y, z0 + kGamma, q, m, half, bad);
            const int t2 = quant_one(xa.z, z0 + 2 * kGamma, q, m, half, bad);
            const int t3 = quant_one(xa.w, z0 + 3 * kGamma, q, m, half, bad);
            i4[g] = make_uchar4((uint8_t)t0, (uint8_t)t1, (uint8_t)t2, (uint8_t)t3);
            count(t0); count(t1); count(t2); count(t3);
        }
        if (two) {
            const uint64_t z0 = seed + (uint64_t)(4 * h + 1) * kGamma;
            const int t0 = quant_one(xb.x, z0, q, m, half, bad), t1 = quant_one(xb.y, z0 + kGamma, q, m, half, bad);
            const int t2 = quant_one(xb.z, z0 + 2 * kGamma, q, m, half, bad);
            const int t3 = quant_one(xb.w, z0 + 3 * kGamma, q, m, half, bad);
            i4[h] = make_uchar4((uint8_t)t0, (uint8_t)t1, (uint8_t)t2, (uint8_t)t3);
            count(t0); count(t1); count(t2); count(t3);
        }
        if (PRIV && (since_fold += 8) >= kFoldEntries) {
            priv_fold(ph, hcount, m);
            since_fold = 0;
        }
    }
    for (int64_t i = 4 * ngroups + g0; i < d; i += stride) {
        const int t = quant_one(x[i], seed + (uint64_t)(i + 1) * kGamma, q, m, half, bad);
        idx[i] = (uint8_t)t;
        count(t);
        if (PRIV && ++since_fold >= kFoldEntries) {
            priv_fold(ph, hcount, m);
            since_fold = 0;
        }
    }
    if (bad) o.st->range_err = 1;
    __syncthreads();
    if (PRIV) {
        // bins of the per-thread counters, summed over the block: warp w takes words w, w + 8, ...
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        for (int w = wid; w < (m + 1) >> 1; w += kQThreads / 32) {
            uint32_t lo = 0, hi = 0;
            for (int c = lane; c < kQThreads; c += 32) {
                const uint32_t v = ph[w * kQThreads + c];
                lo += v & 0xffffu;
                hi += v >> 16;
            }
            for (int o = 16; o; o >>= 1) {
                lo += __shfl_xor_sync(0xffffffffu, lo, o);
                hi += __shfl_xor_sync(0xffffffffu, hi, o);
            }
            if (lane == 0) {
                hcount[2 * w] += lo;  // only warp wid writes these two bins after the barrier
                if (2 * w + 1 < m) hcount[2 * w + 1] += hi;
            }
        }
        __syncthreads();
    }
    for (int r = threadIdx.x; r < m; r += blockDim.x)
        if (hcount[r]) atomicAdd(&o.acc[r], hcount[r]);
    finish_counts(o, m);
}

// ------------------------------------------------ short codebooks (m <= 16)
// The same decisions as k_quantize, and as k_quantize_timeshare with two codebooks (TS), with fewer
// instructions per entry.  What bounds it: instruction issue, 69 instructions an entry in an earlier form and 50 now
// (16 values; issue 76 %), then the pipe for integer logic and compares (63 %).  So
//  * the search takes STEPS = ceil(log2 m) unrolled steps (a template argument); its position is a byte offset
//    that steps by predicated float adds of denormals (bit patterns 4, 8, ..: exact), which the otherwise
//    idle fp32 pipe takes;
//  * the gaps q[t+1] - q[t] are formed once per block; an entry equal to q[t] needs no test of its own (its
//    distance 0 is above no product); the range test is a minimum and a maximum of eight entries, and only a
//    group that fails it looks at its entries one by one;
//  * the draw computes only bits 32..63 of SplitMix64's second product, the bits the
//    rule reads (k = bits 40..63 of the output, and the final xor-shift by 31 leaves
//    bits 40..63 unchanged), with 32-bit limbs: each 64-bit multiply modulo 2^64 is a
//    wide 32 x 32 product plus two 32-bit multiply-adds, and the top word of the second
//    one a high product plus two;
//  * the index counts are per-thread 32-bit counters in shared memory (one column per
//    thread, so the shared-memory adds never meet);
//  * the next eight entries are loaded before this eight's arithmetic.
// 67 million entries, 16 values: 117 us instead of 161 (HBM alone: 49); 16.8 million entries, time-shared
// between two codebooks of 16: 48 instead of 108.
constexpr int kFastBins = 16;
constexpr uint32_t kC1lo = 0x1CE4E5B9u, kC1hi = 0xBF58476Du;  // SplitMix64 multipliers (Steele, Lea, Flood 2014)
constexpr uint32_t kC2lo = 0x133111EBu, kC2hi = 0x94D049BBu;

// Bits 32..63 of the SplitMix64 output for state z = (zh:zl).
__device__ __forceinline__ uint32_t splitmix64_hi(uint32_t zl, uint32_t zh) {
    const uint32_t xl = zl ^ __funnelshift_r(zl, zh, 30), xh = zh ^ (zh >> 30);  // z ^ (z >> 30)
    const uint64_t w = (uint64_t)xl * kC1lo;                                       // (xh:xl) * C1 mod 2^64
    const uint32_t al = (uint32_t)w;
    const uint32_t ah = (uint32_t)(w >> 32) + xl * kC1hi + xh * kC1lo;
    const uint32_t yl = al ^ __funnelshift_r(al, ah, 27), yh = ah ^ (ah >> 27);   // a ^ (a >> 27)
    return __umulhi(yl, kC2lo) + yl * kC2hi + yh * kC2lo;                         // top word of y * C2
}

// 64-bit counter state (zh:zl) advanced by gamma.
__device__ __forceinline__ void add_gamma(uint32_t &zl, uint32_t &zh) {
    const uint64_t z = (((uint64_t)zh << 32) | zl) + kGamma;
    zl = (uint32_t)z;
    zh = (uint32_t)(z >> 32);
}

// TS: entry i takes the second codebook (part 1) iff its draw with seed_ts is below thr (k_quantize_timeshare).
struct ShortArgs {
    const float *x;
    int64_t d;
    const float *Q[2];
    int m[2];
    uint64_t seed, seed_ts;
    uint32_t thr;
    uint8_t *idx, *sel;
};

// (Six blocks an SM, 40 registers: 120 us; four, 52 registers, 133.  Two codebooks: 53 to 57 us either way.)
template <int STEPS, bool TS>
__global__ void __launch_bounds__(kQThreads, TS ? 4 : 6) k_quantize_short(const ShortArgs a, const QuantOut o) {
    constexpr int kParts = TS ? 2 : 1;
    __shared__ float sq[4 * kFastBins];  // thresholds of part 0, of part 1, then the gaps above them
    __shared__ uint32_t ph[kParts * kFastBins * kQThreads];  // ph[t * kQThreads + thread]
    bool wrong = false;
    for (int r = threadIdx.x; r < 2 * kFastBins; r += kQThreads) {
        const int part = r / kFastBins, t = r % kFastBins, m = part ? (TS ? a.m[1] : 0) : a.m[0];
        const float *Q = part ? a.Q[1] : a.Q[0];
        sq[r] = t < m ? Q[t] : CUDART_NAN_F;  // (no entry passes it, +inf neither)
        sq[2 * kFastBins + r] = t + 1 < m ? __fsub_rn(Q[t + 1], Q[t]) : CUDART_INF_F;
        wrong |= t + 1 < m && !(Q[t + 1] > Q[t]);
    }
#pragma unroll
    for (int t = 0; t < kParts * kFastBins; t++) ph[t * kQThreads + threadIdx.x] = 0u;
    const bool unsorted_q = __syncthreads_or(wrong);
    const int64_t d = unsorted_q ? 0 : a.d;  // unsorted: nothing is encoded
    if (unsorted_q && threadIdx.x == 0) o.st->range_err = kUnsortedQ;
    // a group within [lo, hi] is within the range of either codebook; NaN, which no group is within, where a codebook of one
    // value is NaN (a longer one is refused above)
    const float q0[2] = {sq[0], TS && a.m[1] ? sq[kFastBins] : sq[0]};
    const float qm[2] = {sq[a.m[0] - 1], TS && a.m[1] ? sq[kFastBins + a.m[1] - 1] : sq[a.m[0] - 1]};
    float lo = q0[0];
    if (TS) asm("max.NaN.f32 %0, %0, %1;" : "+f"(lo) : "f"(q0[1]));
    const float hi = TS ? fminf(qm[0], qm[1]) : qm[0];
    const char *cq = reinterpret_cast<const char *>(sq);
    char *pc = reinterpret_cast<char *>(ph) + 4 * threadIdx.x;
    constexpr int kTop = STEPS > 0 && !TS;  // the first threshold of the search stays in a register
    const float top = sq[kTop << (STEPS ? STEPS - 1 : 0)];
    bool bad = false;
    // 4 (16 part + index) of an entry with counter states z and zs (TS)
    auto one = [&](float xv, uint32_t zl, uint32_t zh, uint32_t sl, uint32_t sh) -> int {
        float tf = 0.f;  // the byte offset's bits, always a denormal
        if (kTop && top <= xv) tf = __int_as_float(4 << (STEPS - 1));
        if (TS && (splitmix64_hi(sl, sh) >> 8) < a.thr) tf = __int_as_float(4 * kFastBins);
#pragma unroll
        for (int s = STEPS - 1 - kTop; s >= 0; s--)
            if (*reinterpret_cast<const float *>(cq + __float_as_int(tf) + (4 << s)) <= xv)
                tf = __fadd_rn(tf, __int_as_float(4 << s));
        int t = __float_as_int(tf);
        const float qa = *reinterpret_cast<const float *>(cq + t);
        const float gap = *reinterpret_cast<const float *>(cq + t + 8 * kFastBins);
        const float k = __fmul_rn((float)(splitmix64_hi(zl, zh) >> 8), 0x1p-24f);
        if (__fmul_rn(k, gap) < __fsub_rn(xv, qa)) t += 4;
        return t;
    };
    // outside its codebook's range: index 0 and the error flag
    auto checked = [&](float xv, int t) -> int {
        const int part = TS ? t / (4 * kFastBins) : 0;
        if (xv >= (part ? q0[1] : q0[0]) && xv <= (part ? qm[1] : qm[0])) return t;
        bad = true;
        return part * 4 * kFastBins;
    };
    auto add = [&](int t) { atomicAdd(reinterpret_cast<uint32_t *>(pc + t * kQThreads), 1u); };
    const bool vec = ((reinterpret_cast<uintptr_t>(a.x) & 15) == 0) && ((reinterpret_cast<uintptr_t>(a.idx) & 3) == 0) &&
                     (!TS || (reinterpret_cast<uintptr_t>(a.sel) & 3) == 0);
    const int64_t ngroups = vec ? d / 4 : 0;
    const int64_t stride = (int64_t)gridDim.x * kQThreads;
    const int64_t first = (int64_t)blockIdx.x * kQThreads + threadIdx.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(a.x);
    uint32_t *i4 = reinterpret_cast<uint32_t *>(a.idx), *s4 = reinterpret_cast<uint32_t *>(a.sel);
    const float4 none = make_float4(lo, lo, lo, lo);
    float4 na = first < ngroups ? x4[first] : none, nb = first + stride < ngroups ? x4[first + stride] : none;
    for (int64_t g = first; g < ngroups; g += 2 * stride) {
        const int64_t h = g + stride;
        const bool two = h < ngroups;
        const float xs[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
        na = g + 2 * stride < ngroups ? x4[g + 2 * stride] : none;
        nb = h + 2 * stride < ngroups ? x4[h + 2 * stride] : none;
        float mn = xs[0], mx = xs[0];
#pragma unroll
        for (int r = 1; r < 7; r += 2) {
            asm("min.NaN.f32 %0, %0, %1, %2;" : "+f"(mn) : "f"(xs[r]), "f"(xs[r + 1]));
            asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(mx) : "f"(xs[r]), "f"(xs[r + 1]));
        }
        asm("min.NaN.f32 %0, %0, %1;" : "+f"(mn) : "f"(xs[7]));
        asm("max.NaN.f32 %0, %0, %1;" : "+f"(mx) : "f"(xs[7]));
        int ts[8];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t z = a.seed + (uint64_t)(4 * (u ? h : g) + 1) * kGamma;  // entry 4g: seed + (4g + 1) gamma
            const uint64_t zs = a.seed_ts + (uint64_t)(4 * (u ? h : g) + 1) * kGamma;
            uint32_t zl = (uint32_t)z, zh = (uint32_t)(z >> 32), sl = (uint32_t)zs, sh = (uint32_t)(zs >> 32);
#pragma unroll
            for (int r = 0; r < 4; r++) {
                ts[4 * u + r] = one(xs[4 * u + r], zl, zh, sl, sh);
                add_gamma(zl, zh);
                if (TS) add_gamma(sl, sh);
            }
        }
        if (!(mn >= lo && mx <= hi)) {
#pragma unroll
            for (int r = 0; r < 8; r++)
                if (r < 4 || two) ts[r] = checked(xs[r], ts[r]);
        }
        const uint32_t wa = (uint32_t)(ts[0] + (ts[1] << 8) + (ts[2] << 16) + (ts[3] << 24));
        const uint32_t wb = (uint32_t)(ts[4] + (ts[5] << 8) + (ts[6] << 16) + (ts[7] << 24));
        i4[g] = TS ? (wa >> 2) & 0x0F0F0F0Fu : wa >> 2;
        if (TS && a.sel) s4[g] = (wa >> 6) & 0x01010101u;
#pragma unroll
        for (int r = 0; r < 4; r++) add(ts[r]);
        if (two) {
            i4[h] = TS ? (wb >> 2) & 0x0F0F0F0Fu : wb >> 2;
            if (TS && a.sel) s4[h] = (wb >> 6) & 0x01010101u;
#pragma unroll
            for (int r = 4; r < 8; r++) add(ts[r]);
        }
    }
    for (int64_t i = 4 * ngroups + first; i < d; i += stride) {
        const uint64_t z = a.seed + (uint64_t)(i + 1) * kGamma, zs = a.seed_ts + (uint64_t)(i + 1) * kGamma;
        const int t = checked(a.x[i], one(a.x[i], (uint32_t)z, (uint32_t)(z >> 32), (uint32_t)zs, (uint32_t)(zs >> 32)));
        a.idx[i] = (uint8_t)((t >> 2) & (kFastBins - 1));
        if (TS && a.sel) a.sel[i] = (uint8_t)(t / (4 * kFastBins));
        add(t);
    }
    if (bad) o.st->range_err = 1;
    __syncthreads();
    // bin t summed over the block's threads: warp w takes bins w, w + 8, ...
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int t = wid; t < kParts * kFastBins; t += kQThreads / 32) {
        uint32_t c = 0;
        for (int u = lane; u < kQThreads; u += 32) c += ph[t * kQThreads + u];
        c = __reduce_add_sync(0xffffffffu, c);
        // the time-shared counts: the first codebook's, then the second's
        if (lane == 0 && c) atomicAdd(&o.acc[t < kFastBins ? t : a.m[0] + t - kFastBins], c);
    }
    finish_counts(o, a.m[0] + (TS ? a.m[1] : 0));
}

template <bool TS>
static void launch_short(const ShortArgs &a, const QuantOut &o, int steps, unsigned blocks, cudaStream_t st) {
    switch (steps) {
        case 0: k_quantize_short<0, TS><<<blocks, kQThreads, 0, st>>>(a, o); break;
        case 1: k_quantize_short<1, TS><<<blocks, kQThreads, 0, st>>>(a, o); break;
        case 2: k_quantize_short<2, TS><<<blocks, kQThreads, 0, st>>>(a, o); break;
        case 3: k_quantize_short<3, TS><<<blocks, kQThreads, 0, st>>>(a, o); break;
        default: k_quantize_short<4, TS><<<blocks, kQThreads, 0, st>>>(a, o); break;
    }
}
// The search visits q[t + 2^s] for s < ceil(log2 m).
static int search_steps(int m) { return m > 1 ? 32 - __builtin_clz((unsigned)(m - 1)) : 0; }

int launch_quantize(const float *x, int64_t d, const float *Q, int m, uint64_t seed, uint8_t *idx, const QuantOut &o,
                    int num_sms, cudaStream_t stream) {
    const int64_t groups = cdiv(d, 4);
    int64_t blocks = std::min<int64_t>(cdiv(groups, 2 * kQThreads), (int64_t)num_sms * 8);
    if (blocks < 1) blocks = 1;
    note_launch();
    if (m <= kFastBins) {
        const ShortArgs a{x, d, {Q, Q}, {m, 0}, seed, 0, 0, idx, nullptr};
        launch_short<false>(a, o, search_steps(m), (unsigned)blocks, stream);
    } else if (m <= kPrivBins)
        k_quantize<true><<<(unsigned)blocks, kQThreads, 0, stream>>>(x, d, Q, m, seed, idx, o);
    else
        k_quantize<false><<<(unsigned)blocks, kQThreads, 0, stream>>>(x, d, Q, m, seed, idx, o);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

// Two-way time-sharing (Sec. 7): entry i uses Q+ iff k_s * 2^-24 < beta (binary64,
// exact), k_s = top 24 bits of SplitMix64(seed_ts + (i+1) * 0x9E3779B97F4A7C15),
// then rounds within its codebook exactly as k_quantize (seed, same counter i).
// counts: [mm] for Q-, then [mp] for Q+; sel (may be null): 1 where Q+ was used.
__global__ void __launch_bounds__(256) k_quantize_timeshare(const float *__restrict__ x, int64_t d,
                                                            const float *__restrict__ Qm, int mm,
                                                            const float *__restrict__ Qp, int mp, double beta,
                                                            uint64_t seed, uint64_t seed_ts, uint8_t *__restrict__ idx,
                                                            uint8_t *__restrict__ sel, QuantOut o) {
    __shared__ float q[2][kMaxS];
    __shared__ uint32_t hcount[2 * kMaxS];
    // (The order is checked here: with loops of its own for it the encode below compiles to a fifth more time, 535 against
    // 437 us at 67 million entries and 17 or 32 values.)
    bool wrong = false;
    for (int r = threadIdx.x; r < kMaxS; r += blockDim.x) {
        q[0][r] = r < mm ? Qm[r] : CUDART_NAN_F;
        q[1][r] = r < mp ? Qp[r] : CUDART_NAN_F;
        wrong |= r > 0 && ((r < mm && !(Qm[r] > Qm[r - 1])) || (r < mp && !(Qp[r] > Qp[r - 1])));
        hcount[r] = 0;
        hcount[kMaxS + r] = 0;
    }
    if (__syncthreads_or(wrong)) {  // nothing is encoded
        if (threadIdx.x == 0) o.st->range_err = kUnsortedQ;
        d = 0;
    }
    bool bad = false;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += stride) {
        uint64_t zs = splitmix64(seed_ts + (uint64_t)(i + 1) * kGamma);
        int part = __dmul_rn((double)(uint32_t)(zs >> 40), 0x1p-24) < beta ? 1 : 0;
        const int mq = part ? mp : mm;
        int t = quant_one(x[i], seed + (uint64_t)(i + 1) * kGamma, q[part], mq, search_half(mq), bad);
        idx[i] = (uint8_t)t;
        if (sel) sel[i] = (uint8_t)part;
        atomicAdd(&hcount[part * kMaxS + t], 1u);
    }
    if (bad) o.st->range_err = 1;
    __syncthreads();
    for (int r = threadIdx.x; r < mm; r += blockDim.x)
        if (hcount[r]) atomicAdd(&o.acc[r], hcount[r]);
    for (int r = threadIdx.x; r < mp; r += blockDim.x)
        if (hcount[kMaxS + r]) atomicAdd(&o.acc[mm + r], hcount[kMaxS + r]);
    finish_counts(o, mm + mp);
}

int launch_quantize_timeshare(const float *x, int64_t d, const float *Qm, int mm, const float *Qp, int mp,
                              double beta, uint64_t seed, uint64_t seed_ts, uint8_t *idx, uint8_t *sel,
                              const QuantOut &o, int num_sms, cudaStream_t stream) {
    note_launch();
    if (mm <= kFastBins && mp <= kFastBins) {
        const int64_t blocks = std::min<int64_t>(cdiv(cdiv(d, 4), 2 * kQThreads), (int64_t)num_sms * 6);
        // k 2^-24 < beta iff k < ceil(2^24 beta): both products are exact
        const ShortArgs a{x, d, {Qm, Qp}, {mm, mp}, seed, seed_ts, (uint32_t)std::ceil(beta * 16777216.0), idx, sel};
        launch_short<true>(a, o, search_steps(std::max(mm, mp)), (unsigned)blocks, stream);
    } else {
        const int64_t blocks = std::min<int64_t>(cdiv(d, 256), (int64_t)num_sms * 8);
        k_quantize_timeshare<<<(unsigned)blocks, 256, 0, stream>>>(x, d, Qm, mm, Qp, mp, beta, seed, seed_ts, idx, sel, o);
    }
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

}  // namespace ecasq
