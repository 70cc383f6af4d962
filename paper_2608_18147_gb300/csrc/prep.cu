// prep.cu -- step 1 of every solve: sorted copy of x, weighted histogram
// (Sec. 2: "we assume X is sorted ... work with its weighted histogram") and the
// prefix sums N, S, S2 of App. E, accumulated in double-double.
//
// Sort: LSD radix sort, 4 passes of 8 bits over order-preserving uint32 keys
// (-0.0 folded into +0.0).  Each pass: per-block digit counts, one scan of the
// [digit][block] count matrix, and a stable scatter whose in-block ranks come
// from warp match masks.
#include <algorithm>

#include "common.cuh"

namespace ecasq {

__device__ __forceinline__ uint32_t f2key(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key2f(uint32_t k) {
    uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

// The range of the values' last-place exponents u (a value is an integer below 2^24 times 2^u), kept behind
// the status record so that zero means none yet: hi = max u + 200, lo = 200 - min u, over non-zero values.
struct UlpRange { uint32_t hi, lo; };
constexpr size_t kUlpRangeAt = 128;
static_assert(sizeof(DevStatus) <= kUlpRangeAt, "the range lies behind the status record");
__device__ __forceinline__ UlpRange *ulp_range(DevStatus *st) {
    return reinterpret_cast<UlpRange *>(reinterpret_cast<char *>(st) + kUlpRangeAt);
}
__device__ __forceinline__ int ulp_exp(uint32_t bits) { return max((int)((bits >> 23) & 255u), 1) - 150; }
__device__ __forceinline__ void ulp_note(float f, uint32_t &hi, uint32_t &lo) {
    const uint32_t b = __float_as_uint(f);
    if (!(b << 1)) return;
    hi = max(hi, (uint32_t)(ulp_exp(b) + 200));
    lo = max(lo, (uint32_t)(200 - ulp_exp(b)));
}

__global__ void __launch_bounds__(256) k_make_keys(const float *__restrict__ x, int64_t d, uint32_t *__restrict__ keys,
                                                   DevStatus *st) {
    __shared__ uint32_t bhi, blo;
    if (threadIdx.x == 0) bhi = blo = 0u;
    __syncthreads();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint32_t hi = 0u, lo = 0u;
    for (; i < d; i += stride) {
        float f = x[i];
        if (!isfinite(f)) st->nonfinite = 1;
        if (f == 0.0f) f = 0.0f;
        keys[i] = f2key(f);
        ulp_note(f, hi, lo);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_max_sync(0xffffffffu, lo);
    if ((threadIdx.x & 31) == 0) { atomicMax(&bhi, hi); atomicMax(&blo, lo); }
    __syncthreads();
    if (threadIdx.x == 0) { atomicMax(&ulp_range(st)->hi, bhi); atomicMax(&ulp_range(st)->lo, blo); }
}

// counts[digit * nb + block] = number of keys of the block with that digit.
__global__ void __launch_bounds__(256) k_radix_count(const uint32_t *__restrict__ keys, int64_t d, int shift,
                                                     uint32_t *__restrict__ counts, int nb) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int r = 0; r < kSortTile / 256; r++) {
        int64_t i = base + r * 256 + threadIdx.x;
        if (i < d) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    counts[(size_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// In-place exclusive scan of uint32 values.  Block b scans a[b*chunk .. min(n, (b+1)*chunk))
// by 1024 threads, in coalesced tiles of 4096 (four consecutive values per thread) with a
// running carry that starts at carry_in[b] (0 when carry_in is null).  One block with
// chunk = n scans the whole array; with several blocks, carry_in holds the exclusive
// prefix of the chunks' totals (k_scan_chunk_sums, then a one-block scan of those).
__global__ void __launch_bounds__(1024) k_scan_u32(uint32_t *a, int64_t n, int64_t chunk,
                                                   const uint32_t *carry_in) {
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t carry;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = min(n, lo + chunk);
    if (threadIdx.x == 0) carry = carry_in ? carry_in[blockIdx.x] : 0u;
    __syncthreads();
    for (int64_t base = lo; base < hi; base += 4 * 1024) {
        const int64_t i0 = base + 4 * (int64_t)threadIdx.x;
        uint32_t v[4];
#pragma unroll
        for (int e = 0; e < 4; e++) v[e] = i0 + e < hi ? a[i0 + e] : 0u;
        const uint32_t s = v[0] + v[1] + v[2] + v[3];
        uint32_t incl = s;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            uint32_t w = wsum[lane], wi = w;
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += t;
            }
            wsum[lane] = wi - w;
        }
        __syncthreads();
        uint32_t run = carry + wsum[wid] + incl - s;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            if (i0 + e < hi) a[i0 + e] = run;
            run += v[e];
        }
        __syncthreads();  // every thread has read carry and wsum
        if (threadIdx.x == blockDim.x - 1) carry = run;  // the old carry plus this tile's total
        __syncthreads();
    }
}

// Totals of the chunks a[b*chunk .. min(n, (b+1)*chunk)), one block of 1024 per chunk.
__global__ void __launch_bounds__(1024) k_scan_chunk_sums(const uint32_t *__restrict__ a, int64_t n, int64_t chunk,
                                                          uint32_t *__restrict__ sums) {
    __shared__ uint32_t wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = min(n, lo + chunk);
    uint32_t t = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) t += a[i];
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) wsum[wid] = t;
    __syncthreads();
    if (wid == 0) {
        t = wsum[lane];
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) sums[blockIdx.x] = t;
    }
}

// Exclusive scan of the n radix counts: one block while n is small, else the chunks'
// totals, a one-block scan of them and a scan of every chunk from its offset
// (sums: scratch of at least 1024 uint32 values).
static void scan_counts(uint32_t *a, int64_t n, uint32_t *sums, cudaStream_t stream) {
    constexpr int64_t kOneBlock = 1 << 16;
    if (n <= kOneBlock) {
        note_launch();
        k_scan_u32<<<1, 1024, 0, stream>>>(a, n, n, nullptr);
        return;
    }
    const int64_t nchunks = std::min<int64_t>(1024, cdiv(n, 16384));
    const int64_t chunk = cdiv(cdiv(n, nchunks), 4096) * 4096;
    const int64_t nc = cdiv(n, chunk);
    note_launch();
    k_scan_chunk_sums<<<(unsigned)nc, 1024, 0, stream>>>(a, n, chunk, sums);
    note_launch();
    k_scan_u32<<<1, 1024, 0, stream>>>(sums, nc, nc, nullptr);
    note_launch();
    k_scan_u32<<<(unsigned)nc, 1024, 0, stream>>>(a, n, chunk, sums);
}

// Stable scatter of one radix pass.  Warp w of a block takes tile positions w * 256 .. + 255, 32 at a time, so (warp,
// step, lane) is the input order.  A warp ranks its keys against its own digit counters (match masks) with no
// block barrier; after one scan over warps and digits the tile is sorted in shared memory and goes
// out in order, neighbouring keys of a digit to neighbouring words.  (A barrier-bound version, three to a step of
// 256 keys and a word here and there a store: 34 us a pass at 4 million keys, now 26.)
__global__ void __launch_bounds__(256) k_radix_scatter(const uint32_t *__restrict__ kin, uint32_t *__restrict__ kout,
                                                       int64_t d, int shift, const uint32_t *__restrict__ offs,
                                                       int nb) {
    constexpr int kSteps = kSortTile / 256;
    __shared__ uint32_t cnt[8][256];      // keys of the warp with the digit, then where its first goes in the tile
    __shared__ uint32_t go[256];          // global place of a digit's first key less its place in the tile
    __shared__ uint32_t sorted[kSortTile];
    __shared__ uint32_t wsum[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int64_t tbase = (int64_t)blockIdx.x * kSortTile;
    const int n = (int)min((int64_t)kSortTile, d - tbase), w0 = wid * (kSortTile / 8);
    uint32_t key[kSteps], rank[kSteps];
#pragma unroll
    for (int r = 0; r < kSteps; r++) key[r] = w0 + 32 * r + lane < n ? kin[tbase + w0 + 32 * r + lane] : 0u;
    const uint32_t first = offs[(size_t)t * nb + blockIdx.x];
#pragma unroll
    for (int w = 0; w < 8; w++) cnt[w][t] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSteps; r++) {
        const bool valid = w0 + 32 * r + lane < n;
        const uint32_t dig = valid ? (key[r] >> shift) & 255u : 256u + (uint32_t)lane;
        const uint32_t peers = __match_any_sync(0xffffffffu, dig);
        const int lead = __ffs(peers) - 1;
        uint32_t before = 0u;
        if (valid && lane == lead) {
            before = cnt[wid][dig];
            cnt[wid][dig] = before + __popc(peers);
        }
        rank[r] = __shfl_sync(0xffffffffu, before, lead) + __popc(peers & lt_mask);
        __syncwarp();
    }
    __syncthreads();
    // digit t: its keys in the tile, their place there (exclusive scan over the digits), and each warp's part
    uint32_t total = 0u;
#pragma unroll
    for (int w = 0; w < 8; w++) total += cnt[w][t];
    uint32_t incl = total;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    uint32_t at = incl - total;
    for (int w = 0; w < wid; w++) at += wsum[w];
    go[t] = first - at;
#pragma unroll
    for (int w = 0; w < 8; w++) {
        const uint32_t c = cnt[w][t];
        cnt[w][t] = at;
        at += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSteps; r++)
        if (w0 + 32 * r + lane < n) sorted[cnt[wid][(key[r] >> shift) & 255u] + rank[r]] = key[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSteps; r++) {
        const int q = 256 * r + t;
        if (q < n) {
            const uint32_t k = sorted[q];
            kout[go[(k >> shift) & 255u] + (uint32_t)q] = k;
        }
    }
}

// ---------------------------------------------------- prefix sums of x and x^2
// The sums are needed as double-double prefixes.  Where the data's range allows it (exact_window; all but data
// with values 10^-24 of the largest) they are exact integers in units of the smallest last place, 128 bits
// for x and 256 for x^2, rounded once to a double-double: the chip has 2 binary64 operations a cycle and SM, and
// a double-double sum per key in two passes and their block scans took 863 of a preparation's 1240 us at
// d = 4 million (169 now).  A sum that 106 bits hold has the same bits either way.  Else they are
// double-double sums in one fixed order.
template <typename T>
__device__ __forceinline__ T shfl_up(T v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }

// Exact sums of x 2^-B and x^2 2^-2B (two's complement; unsigned), and the number of heads.
struct IntSums {
    uint64_t s[2], q[4];
    int64_t h;
};
// Double-double sums and the number of heads.
struct DDSums { dd s, q; int64_t h; };

__device__ __forceinline__ void add_words(uint64_t (&a)[2], uint64_t b0, uint64_t b1) {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(a[0]), "+l"(a[1]) : "l"(b0), "l"(b1));
}
__device__ __forceinline__ void add_words(uint64_t (&a)[4], uint64_t b0, uint64_t b1, uint64_t b2, uint64_t b3) {
    asm("add.cc.u64 %0, %0, %4;\n\taddc.cc.u64 %1, %1, %5;\n\taddc.cc.u64 %2, %2, %6;\n\taddc.u64 %3, %3, %7;"
        : "+l"(a[0]), "+l"(a[1]), "+l"(a[2]), "+l"(a[3]) : "l"(b0), "l"(b1), "l"(b2), "l"(b3));
}
__device__ __forceinline__ void neg_words(uint64_t (&a)[2]) {
    a[0] = ~a[0];
    a[1] = ~a[1];
    add_words(a, 1, 0);
}

// The top-aligned words of a non-zero integer, and by how many bits it was shifted up.
template <int NW>
__device__ __forceinline__ int align_words(uint64_t (&w)[NW]) {
    int sh = 0;
#pragma unroll
    for (int r = 0; r < NW - 1; r++)
        if (w[NW - 1] == 0) {
#pragma unroll
            for (int i = NW - 1; i > 0; i--) w[i] = w[i - 1];
            w[0] = 0;
            sh += 64;
        }
    const int c = __clzll((long long)w[NW - 1]);
    if (c) {
#pragma unroll
        for (int i = NW - 1; i > 0; i--) w[i] = w[i] << c | w[i - 1] >> (64 - c);
        w[0] <<= c;
    }
    return sh + c;
}
// The double nearest to w 2^e, ties to even (w non-zero; in the normal range); w becomes the distance to it,
// rounded_up its direction.
template <int NW>
__device__ __forceinline__ double take_double(uint64_t (&w)[NW], int e, bool neg, bool &rounded_up, int &e_out) {
    e -= align_words(w);
    uint64_t m = w[NW - 1] >> 11, rest = w[NW - 1] & 0x7FFu, low = 0;
#pragma unroll
    for (int i = 0; i < NW - 1; i++) low |= w[i];
    rounded_up = rest > 0x400u || (rest == 0x400u && (low != 0 || (m & 1u)));
    w[NW - 1] = rest;
    if (rounded_up) {  // the distance is 2^(64 NW - 53) - rest
        m++;
        uint64_t carry = 1;
#pragma unroll
        for (int i = 0; i < NW; i++) {
            w[i] = ~w[i] + carry;
            carry = carry && w[i] == 0;
        }
        w[NW - 1] &= 0x7FFu;
    }
    e_out = e;
    int x = e + 64 * NW - 53 + 52 + 1023;
    if (m >> 53) { m >>= 1; x++; }
    return __longlong_as_double((long long)((neg ? 1ull << 63 : 0ull) | (uint64_t)x << 52 | (m & ((1ull << 52) - 1))));
}
// w 2^e (negated if neg) as the double-double nearest to it.
template <int NW>
__device__ __forceinline__ dd words_to_dd(uint64_t (&w)[NW], int e, bool neg) {
    uint64_t any = 0;
#pragma unroll
    for (int i = 0; i < NW; i++) any |= w[i];
    if (!any) return {0.0, 0.0};
    bool up, up2;
    int e1, e2;
    const double hi = take_double(w, e, neg, up, e1);
    any = 0;
#pragma unroll
    for (int i = 0; i < NW; i++) any |= w[i];
    if (!any) return {hi, 0.0};
    return {hi, take_double(w, e1, neg != up, up2, e2)};
}

// How a data set is summed: B < kNoWindow, exact integers in units of 2^B.
constexpr int kNoWindow = 1 << 20;
__device__ __forceinline__ int exact_window(UlpRange r, int64_t d) {
    if (!r.hi) return 0;  // zeros only
    const int umin = 200 - (int)r.lo, umax = (int)r.hi - 200, bits = 64 - __clzll(d);
    return 24 + umax - umin + bits <= 126 ? umin : kNoWindow;  // x^2: 48 + 2 (umax - umin) + bits <= 252
}

struct SumInt {
    using Val = IntSums;
    int B;
    __device__ Val zero() const { return {{0, 0}, {0, 0, 0, 0}, 0}; }
    __device__ void add_key(Val &a, uint32_t key) const {
        const uint32_t b = __float_as_uint(key2f(key));
        const uint32_t m = (b & 0x7FFFFFu) | (b & 0x7F800000u ? 0x800000u : 0u);
        const int sh = m ? ulp_exp(b) - B : 0;
        const uint64_t v = m;
        uint64_t x[2] = {sh < 64 ? v << sh : 0ull, sh < 64 ? (sh ? v >> (64 - sh) : 0ull) : v << (sh - 64)};
        if (b >> 31) neg_words(x);
        add_words(a.s, x[0], x[1]);
        const uint64_t q = v * v;
        const int w = 2 * sh >> 6, c = 2 * sh & 63;
        const uint64_t l = q << c, h = c ? q >> (64 - c) : 0ull;
        add_words(a.q, w == 0 ? l : 0ull, w == 1 ? l : w == 0 ? h : 0ull, w == 2 ? l : w == 1 ? h : 0ull,
                  w == 3 ? l : w == 2 ? h : 0ull);
    }
    __device__ Val add(const Val &a, const Val &b) const {
        Val r = a;
        add_words(r.s, b.s[0], b.s[1]);
        add_words(r.q, b.q[0], b.q[1], b.q[2], b.q[3]);
        r.h += b.h;
        return r;
    }
    // a - b (b summed into a before)
    __device__ Val sub(const Val &a, const Val &b) const {
        Val r = a;
        asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;" : "+l"(r.s[0]), "+l"(r.s[1]) : "l"(b.s[0]), "l"(b.s[1]));
        asm("sub.cc.u64 %0, %0, %4;\n\tsubc.cc.u64 %1, %1, %5;\n\tsubc.cc.u64 %2, %2, %6;\n\tsubc.u64 %3, %3, %7;"
            : "+l"(r.q[0]), "+l"(r.q[1]), "+l"(r.q[2]), "+l"(r.q[3]) : "l"(b.q[0]), "l"(b.q[1]), "l"(b.q[2]), "l"(b.q[3]));
        r.h -= b.h;
        return r;
    }
    __device__ Val shfl_up(const Val &v, int o) const {
        Val t;
#pragma unroll
        for (int i = 0; i < 2; i++) t.s[i] = ecasq::shfl_up(v.s[i], o);
#pragma unroll
        for (int i = 0; i < 4; i++) t.q[i] = ecasq::shfl_up(v.q[i], o);
        t.h = ecasq::shfl_up(v.h, o);
        return t;
    }
    __device__ dd s_of(const Val &v) const {
        uint64_t w[2] = {v.s[0], v.s[1]};
        const bool neg = w[1] >> 63;
        if (neg) neg_words(w);
        return words_to_dd(w, B, neg);
    }
    __device__ dd q_of(const Val &v) const {
        uint64_t w[4] = {v.q[0], v.q[1], v.q[2], v.q[3]};
        return words_to_dd(w, 2 * B, false);
    }
};

// x^2 of a binary32 value is exact in binary64.
struct SumDD {
    using Val = DDSums;
    __device__ Val zero() const { return {{0.0, 0.0}, {0.0, 0.0}, 0}; }
    __device__ void add_key(Val &a, uint32_t key) const {
        const double x = (double)key2f(key);
        a.s = dd_add_d(a.s, x);
        a.q = dd_add_d(a.q, __dmul_rn(x, x));
    }
    __device__ Val add(const Val &a, const Val &b) const { return {dd_add(a.s, b.s), dd_add(a.q, b.q), a.h + b.h}; }
    __device__ Val sub(const Val &a, const Val &b) const { return {dd_sub(a.s, b.s), dd_sub(a.q, b.q), a.h - b.h}; }
    __device__ Val shfl_up(const Val &v, int o) const {
        return {{ecasq::shfl_up(v.s.hi, o), ecasq::shfl_up(v.s.lo, o)}, {ecasq::shfl_up(v.q.hi, o), ecasq::shfl_up(v.q.lo, o)},
                ecasq::shfl_up(v.h, o)};
    }
    __device__ dd s_of(const Val &v) const { return v.s; }
    __device__ dd q_of(const Val &v) const { return v.q; }
};
// One tile's partial of either kind.
union HistPart { IntSums i; DDSums d; };
static_assert(sizeof(HistPart) <= 192, "a tile of kHistTile keys has four scan tiles' room");
__device__ __forceinline__ IntSums &part_of(HistPart &p, const SumInt &) { return p.i; }
__device__ __forceinline__ DDSums &part_of(HistPart &p, const SumDD &) { return p.d; }

// Block-wide inclusive scan of one value per thread (256 threads).
template <typename Sum>
__device__ typename Sum::Val block_scan_incl(const Sum &sum, typename Sum::Val v, HistPart *wtot, typename Sum::Val &total) {
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const typename Sum::Val t = sum.shfl_up(v, o);
        if (lane >= o) v = sum.add(t, v);
    }
    if (lane == 31) part_of(wtot[wid], sum) = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        typename Sum::Val acc = part_of(wtot[0], sum);
        for (int w = 1; w < 8; w++) { acc = sum.add(acc, part_of(wtot[w], sum)); part_of(wtot[w], sum) = acc; }
    }
    __syncthreads();
    if (wid > 0) v = sum.add(part_of(wtot[wid - 1], sum), v);
    total = part_of(wtot[7], sum);
    __syncthreads();
    return v;
}

// The thread's kHistPer consecutive sorted keys starting at base (positions >= d are left out): the sums of x and
// x^2 and the number of heads.  One fixed order per thread, so the single-row and the batched
// paths, which both call it, give the same bits.
template <typename Sum>
__device__ __forceinline__ typename Sum::Val hist_thread_sums(const Sum &sum, const uint32_t *keys, int64_t d, int64_t base) {
    typename Sum::Val v = sum.zero();
    uint32_t prev = base > 0 && base - 1 < d ? keys[base - 1] : 0u;
#pragma unroll 4
    for (int e = 0; e < kHistPer; e++) {
        const int64_t i = base + e;
        if (i < d) {
            const uint32_t k = keys[i];
            sum.add_key(v, k);
            v.h += (i == 0 || k != prev) ? 1 : 0;
            prev = k;
        }
    }
    return v;
}

// Pass C for the thread's keys: from the exclusive prefix `run` before them, every head
// i writes its unique index u = run.h, v[u], N[u] = i, S[u] and S2[u] (hi at [u], lo at
// [lo_off + u]); the last position d - 1 also writes the totals at index p and returns
// p and ||X||^2 through p_out and norm2_out.
template <typename Sum>
__device__ __forceinline__ void hist_thread_fill(const Sum &sum, const uint32_t *keys, int64_t d, int64_t base,
                                                 typename Sum::Val run, float *v, int64_t *N, double *S, double *S2,
                                                 int64_t lo_off, int64_t *p_out, double *norm2_out) {
    uint32_t prev = base > 0 && base - 1 < d ? keys[base - 1] : 0u;
#pragma unroll 1
    for (int e = 0; e < kHistPer; e++) {
        const int64_t i = base + e;
        if (i >= d) break;
        const uint32_t k = keys[i];
        const bool head = i == 0 || k != prev;
        prev = k;
        if (head) {
            const int64_t u = run.h;
            const dd ss = sum.s_of(run), qq = sum.q_of(run);
            v[u] = key2f(k);
            N[u] = i;
            S[u] = ss.hi; S[lo_off + u] = ss.lo;
            S2[u] = qq.hi; S2[lo_off + u] = qq.lo;
        }
        sum.add_key(run, k);
        run.h += head ? 1 : 0;
        if (i == d - 1) {
            const int64_t p = run.h;
            const dd ss = sum.s_of(run), qq = sum.q_of(run);
            N[p] = d;
            S[p] = ss.hi; S[lo_off + p] = ss.lo;
            S2[p] = qq.hi; S2[lo_off + p] = qq.lo;
            *p_out = p;
            *norm2_out = qq.hi;
        }
    }
}

// Pass C of a whole tile of kHistTile keys by exact sums: a warp takes 512 consecutive keys, 32 at a time, a lane
// one, so that neighbouring heads' results are neighbouring stores.  (Sixteen consecutive keys a thread wrote
// every value to a sector of its own: 186 us at 4 million values, now 136.)  Integer sums do not depend on
// their order, so the results are hist_thread_fill's.
__device__ __forceinline__ void hist_tile_fill(const SumInt &sum, const uint32_t *keys, int64_t d, const IntSums &before,
                                               HistPart *wtot, float *v, int64_t *N, double *S, double *S2, int64_t lo_off,
                                               int64_t *p_out, double *norm2_out) {
    constexpr int kPerWarp = kHistTile / 8;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kHistTile + wid * kPerWarp;
    IntSums t = sum.zero();
#pragma unroll 4
    for (int e = 0; e < kPerWarp; e += 32) {
        const int64_t i = base + e + lane;
        if (i >= d) continue;
        const uint32_t k = keys[i];
        sum.add_key(t, k);
        t.h += (i == 0 || k != keys[i - 1]) ? 1 : 0;
    }
    for (int o = 16; o; o >>= 1) {
        IntSums x;
#pragma unroll
        for (int r = 0; r < 2; r++) x.s[r] = __shfl_xor_sync(full, t.s[r], o);
#pragma unroll
        for (int r = 0; r < 4; r++) x.q[r] = __shfl_xor_sync(full, t.q[r], o);
        x.h = __shfl_xor_sync(full, t.h, o);
        t = sum.add(t, x);
    }
    if (lane == 0) wtot[wid].i = t;
    __syncthreads();
    IntSums run = before;  // the sums before the warp's next 32 keys
    for (int w = 0; w < wid; w++) run = sum.add(run, wtot[w].i);
#pragma unroll 1
    for (int e = 0; e < kPerWarp; e += 32) {
        const int64_t i = base + e + lane;
        if (base + e >= d) break;  // warp-uniform
        const uint32_t k = i < d ? keys[i] : 0u;
        const bool head = i < d && (i == 0 || k != keys[i - 1]);
        const unsigned heads = __ballot_sync(full, head);
        IntSums x = sum.zero();
        if (i < d) sum.add_key(x, k);
        IntSums incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            const IntSums y = sum.shfl_up(incl, o);
            if (lane >= o) incl = sum.add(y, incl);
        }
        incl = sum.add(run, incl);
        if (head) {
            const IntSums at = sum.sub(incl, x);
            const int64_t u = run.h + __popc(heads & ((1u << lane) - 1u));
            const dd ss = sum.s_of(at), qq = sum.q_of(at);
            v[u] = key2f(k);
            N[u] = i;
            S[u] = ss.hi; S[lo_off + u] = ss.lo;
            S2[u] = qq.hi; S2[lo_off + u] = qq.lo;
        }
        const int64_t h = run.h + __popc(heads);
        if (i == d - 1) {
            const dd ss = sum.s_of(incl), qq = sum.q_of(incl);
            N[h] = d;
            S[h] = ss.hi; S[lo_off + h] = ss.lo;
            S2[h] = qq.hi; S2[lo_off + h] = qq.lo;
            *p_out = h;
            *norm2_out = qq.hi;
        }
#pragma unroll
        for (int r = 0; r < 2; r++) run.s[r] = __shfl_sync(full, incl.s[r], 31);
#pragma unroll
        for (int r = 0; r < 4; r++) run.q[r] = __shfl_sync(full, incl.q[r], 31);
        run.h = h;
    }
}

// f(sum) with the data set's way of summing.
template <typename F>
__device__ __forceinline__ void with_sums(UlpRange r, int64_t d, F &&f) {
    const int B = exact_window(r, d);
    if (B < kNoWindow) f(SumInt{B});
    else f(SumDD{});
}

// Pass A of the histogram scan: per tile of kHistTile sorted keys, the number of unique-value heads and the sums
// of x and x^2.
__global__ void __launch_bounds__(256) k_hist_partials(const uint32_t *__restrict__ keys, int64_t d, HistPart *part,
                                                       DevStatus *st) {
    __shared__ HistPart wtot[8];
    with_sums(*ulp_range(st), d, [&](auto sum) {
        const auto v = hist_thread_sums(sum, keys, d, (int64_t)blockIdx.x * kHistTile + (int64_t)threadIdx.x * kHistPer);
        auto tot = v;
        block_scan_incl(sum, v, wtot, tot);
        if (threadIdx.x == 0) part_of(part[blockIdx.x], sum) = tot;
    });
}

// Exclusive scan of the tiles' partials by one block of 256 threads: each thread sums a
// contiguous run of tiles in order, the runs' totals are scanned across the block
// (block_scan_incl), and each thread then writes its run's exclusive prefixes.
__global__ void __launch_bounds__(256) k_hist_scan_partials(HistPart *part, int64_t nb, int64_t d, DevStatus *st) {
    __shared__ HistPart wtot[8];
    __shared__ HistPart incl_all[256];
    const int64_t per = cdiv(nb, (int64_t)blockDim.x);
    const int64_t lo = min((int64_t)threadIdx.x * per, nb), hi = min(lo + per, nb);
    with_sums(*ulp_range(st), d, [&](auto sum) {
        auto s = sum.zero();
        for (int64_t b = lo; b < hi; b++) s = sum.add(s, part_of(part[b], sum));
        auto total = s;
        part_of(incl_all[threadIdx.x], sum) = block_scan_incl(sum, s, wtot, total);
        if (threadIdx.x == 0) st->p = total.h;
        __syncthreads();
        auto acc = threadIdx.x > 0 ? part_of(incl_all[threadIdx.x - 1], sum) : sum.zero();
        for (int64_t b = lo; b < hi; b++) {
            const auto t = part_of(part[b], sum);
            part_of(part[b], sum) = acc;
            acc = sum.add(acc, t);
        }
    });
}

// Pass C: per sorted position i that starts a run of equal keys (a head), the
// unique index u and v[u], N[u] = i, S[u], S2[u] (exclusive prefix sums).
// The last position also writes N[p] = d, S[p], S2[p] and ||X||^2.  S and S2 hold hi[0..p], then lo[0..p].
__global__ void __launch_bounds__(256) k_hist_fill(const uint32_t *__restrict__ keys, int64_t d, HistPart *part,
                                                   float *v, int64_t *N, double *S, double *S2, DevStatus *st) {
    __shared__ HistPart wtot[8];
    const int64_t base = (int64_t)blockIdx.x * kHistTile + (int64_t)threadIdx.x * kHistPer;
    const int64_t lo_off = *(volatile int64_t *)&st->p + 1;  // the number of unique values: k_hist_scan_partials
    int64_t p;  // (the same again)
    const int B = exact_window(*ulp_range(st), d);
    if (B < kNoWindow) {
        hist_tile_fill(SumInt{B}, keys, d, part[blockIdx.x].i, wtot, v, N, S, S2, lo_off, &p, &st->norm2);
        return;
    }
    {
        const SumDD sum;
        const auto loc = hist_thread_sums(sum, keys, d, base);
        auto tot = loc;
        const auto incl = block_scan_incl(sum, loc, wtot, tot);
        // exclusive prefix before this thread's first element
        const auto run = sum.add(part_of(part[blockIdx.x], sum), sum.sub(incl, loc));
        hist_thread_fill(sum, keys, d, base, run, v, N, S, S2, lo_off, &p, &st->norm2);
    }
}

__global__ void k_hist_weights(const int64_t *N, int64_t *w, const DevStatus *st) {
    const int64_t p = st->p, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += stride) w[i] = N[i + 1] - N[i];
}

// ------------------------------------------------------------ short rows
// One block per row of length d <= kScanTile: the sorted keys (bitonic sort in
// shared memory; the order is unique, so any exact sort gives the same keys) and
// then the arithmetic of k_hist_fill for a single tile (zero tile offset), so that
// v, w, N, S, S2, p and ||X||^2 of every row equal what prepare_device gives for
// that row alone.
// st, where given: the status record, which starts at zero.
__global__ void __launch_bounds__(256) k_rows_prepare(const float *__restrict__ X, RowsData R, DevStatus *st) {
    if (st && blockIdx.x == 0 && threadIdx.x < sizeof(DevStatus) / 8) reinterpret_cast<int64_t *>(st)[threadIdx.x] = 0;
    __shared__ uint32_t keys[kScanTile];
    __shared__ HistPart wtot[8];
    __shared__ int nonfin;
    __shared__ UlpRange range;
    const int64_t row = blockIdx.x;
    const int d = (int)R.d;
    const float *x = X + row * R.d;
    if (threadIdx.x == 0) {
        nonfin = 0;
        range = {0u, 0u};
    }
    __syncthreads();
    uint32_t hi = 0u, lo = 0u;
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        uint32_t k = 0xFFFFFFFFu;  // above every finite key: padding sorts last
        if (i < d) {
            float f = x[i];
            if (!isfinite(f)) nonfin = 1;
            if (f == 0.0f) f = 0.0f;
            k = f2key(f);
            ulp_note(f, hi, lo);
        }
        keys[i] = k;
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_max_sync(0xffffffffu, lo);
    if ((threadIdx.x & 31) == 0) { atomicMax(&range.hi, hi); atomicMax(&range.lo, lo); }
    __syncthreads();
    int n2 = 1;
    while (n2 < d) n2 <<= 1;
    for (int kk = 2; kk <= n2; kk <<= 1) {
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                int l = i ^ jj;
                if (l > i) {
                    uint32_t a = keys[i], b = keys[l];
                    bool up = (i & kk) == 0;
                    if ((a > b) == up) { keys[i] = b; keys[l] = a; }
                }
            }
            __syncthreads();
        }
    }
    const int64_t dcap = R.dcap;
    float *v = R.v + row * dcap;
    int64_t *N = R.N + row * (dcap + 1), *w = R.w + row * dcap;
    double *S = R.S + row * 2 * (dcap + 1), *S2 = R.S2 + row * 2 * (dcap + 1);
    // k_hist_fill, one tile
    const int64_t base = (int64_t)threadIdx.x * kHistPer;
    __shared__ int64_t p_sm;
    with_sums(range, d, [&](auto sum) {
        const auto loc = hist_thread_sums(sum, keys, d, base);
        auto tot = loc;
        const auto incl = block_scan_incl(sum, loc, wtot, tot);
        const auto run = sum.add(sum.zero(), sum.sub(incl, loc));
        hist_thread_fill(sum, keys, d, base, run, v, N, S, S2, tot.h + 1, R.p + row, R.norm2 + row);
        if (threadIdx.x == 0) p_sm = tot.h;
    });
    __syncthreads();
    const int64_t p = p_sm;
    for (int u = threadIdx.x; u < p; u += blockDim.x) w[u] = N[u + 1] - N[u];
    if (threadIdx.x == 0) R.nonfinite[row] = nonfin;
}

__global__ void k_rows_finite(const float *__restrict__ x, int64_t n, DevStatus *st) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) bad |= !isfinite(x[i]);
    if (bad) st->nonfinite = 1;
}

// Raises st->nonfinite when one of the n values is not finite.
int launch_rows_finite(const float *x, int64_t n, DevStatus *ds, cudaStream_t st) {
    note_launch();
    k_rows_finite<<<(unsigned)std::min<int64_t>(cdiv(n, 256), 4096), 256, 0, st>>>(x, n, ds);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

int launch_rows_prepare(const float *X, int64_t rows, const RowsData &R, DevStatus *ds, cudaStream_t st) {
    if (R.d < 1 || R.d > kScanTile) return ECASQ_EINVAL;
    note_launch();
    static_assert(sizeof(DevStatus) % 8 == 0, "cleared by 64-bit words");
    k_rows_prepare<<<(unsigned)rows, 256, 0, st>>>(X, R, ds);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

// ------------------------------------------------------------ general P
// The histogram view over a caller-given candidate set P (Sec. 5, App. E): for
// every grid point t, u_t = #{unique x <= p_t}; N, S, S2 at t+1 are the unique-value
// prefix sums at u_t (the sums of all entries x <= p_t), so w_t = #{p_(t-1) < x <= p_t}.
// Flags st->range_err when P is not strictly ascending and finite, starts above min x
// or ends below max x (App. E: then no quantizer drawn from P spans X), and records
// the sizes of the first- and last-value sets L = {a : p_a <= min x} and
// R = {b : p_b >= max x} of eqs. apx_base and apx_final in st->grid_nL, grid_nR.
// vX, NX, SX, S2X: the unique-value arrays (pX values, packed hi | lo).
__global__ void k_grid_prefix(const float *__restrict__ P, int64_t n, const float *__restrict__ vX,
                              const int64_t *__restrict__ NX, const double *__restrict__ SX,
                              const double *__restrict__ S2X, int64_t pX, float *v, int64_t *w, int64_t *N, double *S,
                              double *S2, DevStatus *st) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
        float pt = P[t];
        if (pt == 0.0f) pt = 0.0f;
        bool bad = !isfinite(pt);
        if (t > 0 && !(P[t] > P[t - 1])) bad = true;
        if (t == 0 && !(pt <= vX[0])) bad = true;
        if (t == n - 1 && !(pt >= vX[pX - 1])) bad = true;
        if (bad) st->range_err = 1;
        // L = {a : p_a <= min x} and R = {b : p_b >= max x} are runs at the two ends
        // (P ascending): the last member of L and the first of R record the sizes
        if (pt <= vX[0] && (t == n - 1 || !(P[t + 1] <= vX[0]))) st->grid_nL = t + 1;
        if (pt >= vX[pX - 1] && (t == 0 || !(P[t - 1] >= vX[pX - 1]))) st->grid_nR = n - t;
        // u = #{unique values <= pt} (binary search)
        int64_t lo = 0, hi = pX;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (vX[mid] <= pt) lo = mid + 1; else hi = mid;
        }
        v[t] = pt;
        N[t + 1] = NX[lo];
        S[t + 1] = SX[lo]; S[n + 1 + t + 1] = SX[pX + 1 + lo];
        S2[t + 1] = S2X[lo]; S2[n + 1 + t + 1] = S2X[pX + 1 + lo];
        if (t == 0) { N[0] = 0; S[0] = 0.0; S[n + 1] = 0.0; S2[0] = 0.0; S2[n + 1] = 0.0; }
    }
}

__global__ void k_grid_weights(const int64_t *N, int64_t n, int64_t *w) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) w[t] = N[t + 1] - N[t];
}

int launch_grid_prefix(const float *P, int64_t n, const float *vX, const int64_t *NX, const double *SX,
                       const double *S2X, int64_t pX, float *v, int64_t *w, int64_t *N, double *S, double *S2,
                       DevStatus *st, cudaStream_t stream) {
    const unsigned blocks = (unsigned)std::min<int64_t>(cdiv(n, 256), 4096);
    note_launch();
    k_grid_prefix<<<blocks, 256, 0, stream>>>(P, n, vX, NX, SX, S2X, pX, v, w, N, S, S2, st);
    ECASQ_LAUNCH_CHECK();
    note_launch();
    k_grid_weights<<<blocks, 256, 0, stream>>>(N, n, w);
    ECASQ_LAUNCH_CHECK();
    return ECASQ_OK;
}

int prepare_device(const float *x, int64_t d, void *ws, const Layout &L, cudaStream_t stream, int64_t *p_host,
                   double *norm2_host) {
    DevStatus *st = wsp<DevStatus>(ws, L.status);
    uint32_t *k0 = wsp<uint32_t>(ws, L.keys0), *k1 = wsp<uint32_t>(ws, L.keys1);
    uint32_t *cnt = wsp<uint32_t>(ws, L.rcount);
    ECASQ_CUDA_TRY(cudaMemsetAsync(st, 0, kUlpRangeAt + sizeof(UlpRange), stream));
    int nb = (int)cdiv(d, kSortTile);
    note_launch();
    k_make_keys<<<(unsigned)std::min<int64_t>(cdiv(d, 256), 4096), 256, 0, stream>>>(x, d, k0, st);
    ECASQ_LAUNCH_CHECK();
    uint32_t *a = k0, *b = k1;
    for (int shift = 0; shift < 32; shift += 8) {
        note_launch();
        k_radix_count<<<nb, 256, 0, stream>>>(a, d, shift, cnt, nb);
        scan_counts(cnt, (int64_t)256 * nb, wsp<uint32_t>(ws, L.v), stream);  // v is free until the histogram
        note_launch();
        k_radix_scatter<<<nb, 256, 0, stream>>>(a, b, d, shift, cnt, nb);
        ECASQ_LAUNCH_CHECK();
        uint32_t *t = a; a = b; b = t;
    }
    // a == k0 holds the sorted keys
    int64_t nbs = cdiv(d, kHistTile);  // the layout holds cdiv(d, kScanTile) >= nbs partials
    HistPart *part = wsp<HistPart>(ws, L.part);
    note_launch();
    k_hist_partials<<<(unsigned)nbs, 256, 0, stream>>>(a, d, part, st);
    note_launch();
    k_hist_scan_partials<<<1, 256, 0, stream>>>(part, nbs, d, st);
    note_launch();
    k_hist_fill<<<(unsigned)nbs, 256, 0, stream>>>(a, d, part, wsp<float>(ws, L.v), wsp<int64_t>(ws, L.N),
                                                 wsp<double>(ws, L.S), wsp<double>(ws, L.S2), st);
    ECASQ_LAUNCH_CHECK();
    note_launch();
    k_hist_weights<<<(unsigned)std::min<int64_t>(cdiv(d + 1, 256), 4096), 256, 0, stream>>>(
        wsp<int64_t>(ws, L.N), wsp<int64_t>(ws, L.w), st);
    ECASQ_LAUNCH_CHECK();
    DevStatus h;
    ECASQ_CUDA_TRY(cudaMemcpyAsync(&h, st, sizeof(DevStatus), cudaMemcpyDeviceToHost, stream));
    ECASQ_CUDA_TRY(cudaStreamSynchronize(stream));
    if (h.nonfinite) return ECASQ_ENONFINITE;
    *p_host = h.p;
    *norm2_host = h.norm2;
    return ECASQ_OK;
}

}  // namespace ecasq
