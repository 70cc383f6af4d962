// dp_fast.cu -- fast approximate DP (Sec. 5, eqs. apx_base / apx_rec / apx_final).
//
// Three stages per DP pass, for up to 8 multipliers at once:
//
// 1. k_wavefront: an fp32 filter over the whole (k, j) triangle with every layer
//    i = 3..s in one cooperative launch, one persistent CTA per SM, in panels of 15
//    column blocks of 64 (the phases are described at `panels` below).  The interval
//    costs C[k,j] and Phi[k,j] of a 64 x 64 tile (App. E quantities rebuilt with
//    compensated fp32 recurrences that add one point at a time, all terms
//    non-negative, from a double-double anchor per tile and column) come from a
//    table built once per call (ECASQ_RESIDENT_COSTS), from a bounded buffer that
//    holds a band of column blocks (ECASQ_STREAMED_COSTS), or are built by the kernel
//    itself a panel at a time; the values are bit-identical.  Per output the kernel
//    keeps the fp32 minimum and up to two runs of tiles whose minimum came within the
//    certified error band of it.
// 2. k_need_layer (layers s down to 3): the outputs whose exact value the
//    answer depends on.  eq. apx_final needs dp(i, p-1) for every i; an output
//    resolved exactly needs the exact values of its band members in the layer
//    below.  For every needed output the kernel re-evaluates its listed tiles
//    (within the certified bound; bit-identically from the resident table), keeps the members k whose fp32 value lies within the
//    band (up to 8 inline, the count either way) and marks (i-1, k) needed.
//    With ECASQ_EXACT_TABLES every output is needed.
// 3. k_exact_layer (layers 3 up to s, over the lists the need
//    stage wrote; k_fill_unneeded first): re-score the members of every needed
//    output in binary64 with double-double interval costs (the reference
//    formulas) and take the lowest k among exact minima: dp64, bp.  Outputs
//    with more members re-scan their band's tiles in fp32 and re-score the
//    members they meet on the fly -- never a full binary64 scan.  Outputs not
//    needed keep their fp32 minimum (dp64 = m32, bp = -2).
//
// The fp32 band: with u = 2^-24, each fp32 candidate value carries a relative
// error of at most eps_i = max(eps_{i-1}, 24u) + 1.0001u (eps_2 = 1.0001u), so
// the exact argmin k* satisfies val32(k*) <= m32 (1 + eps_i)/(1 - eps_i) for
// ANY fp32 evaluation within that bound (the re-evaluations of stages 2 and 3
// need not be bit-identical to the wavefront's).  The 24u budget for one
// interval cost (about 21u used): column anchors within 2u (C: 4.5u) from a
// double-double corner and compensated scans of non-negative increments,
// compensated recurrences of non-negative point terms, correctly rounded
// reciprocal and products, and the documented error of __log2f (2^-22
// absolute on [0.5,2), 2 ulp elsewhere) amplified at most 2.44x through
// h(y) = -y log2 y for y <= 1/2; values y > 1/2 are evaluated through 1 - y
// computed from the complementary mass.  The exact stage re-checks
// |m32 - dp64| <= eps_i dp64 for every resolved output and counts violations.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "cost32.cuh"

namespace ecasq {

int launch_dp_reference(const Prefix &P, const double *lamp, int G, int s, double *dp64, int32_t *bp,
                        cudaStream_t st);
void timer_begin(cudaStream_t st);
void timer_end(cudaStream_t st);

constexpr int BJ = 64;         // columns per block
constexpr int BK = 64;         // k per tile
constexpr int NPROD = 64;      // threads that build a cost tile: one per column of the block
constexpr int kTaskWords = 4;  // far tasks of a multiplier split: at most 32 of these words
constexpr int PSTR = BK + 4;   // padded row stride (floats) of the interval-cost buffers
constexpr int MAXCONS = 512;   // threads of a wavefront CTA: every phase is latency-bound at 256
constexpr int NMEM = 8;        // members kept inline per output
constexpr int64_t kMaxFastP = (int64_t)1 << 20;
constexpr uint32_t kSpinLimit = 1u << 26;
constexpr uint32_t kTestSpinLimit = 1u << 14;  // the ECASQ_TEST_STALL hook: about 10-20 ms of spinning
constexpr uint32_t kCopySpinLimit = 1u << 22;  // waits on bulk copies (microseconds when healthy)
// Resident interval costs: per tile, C[64][PSTR] then Phi[64][PSTR] (the shared-memory layout).
constexpr int kCostHalfFloats = BJ * PSTR;
constexpr uint32_t kCostHalfBytes = (uint32_t)(kCostHalfFloats * sizeof(float));  // 17408, a multiple of 16
constexpr size_t kCostTileFloats = 2 * (size_t)kCostHalfFloats;

// Band of an output: up to two runs of tile indices K (< 2^14), tiles appended in
// increasing K (fold_panel).  Low word: run 1 as first << 16 | last; high word: run 2 the same way,
// 0 when absent (a second run starts at a tile >= 2).  A tile within the band opens run 1,
// or extends it when it follows run 1 directly and there is no run 2, else opens run 2, else
// extends run 2 to itself (the gap is then scanned too: a superset, never a miss).  A tile
// below the band restarts it: run 1 = [K, K], no run 2.
__device__ __forceinline__ uint64_t band_pack(uint32_t w1, uint32_t w2) { return ((uint64_t)w2 << 32) | w1; }

// Per-pass constants, copied once to device memory (kernels index them at run time).
struct FastParams {
    float tau[kMaxS + 1];  // per layer: band factor 2 eps_i / (1 - eps_i), with margin
    float eps[kMaxS + 1];  // per layer: eps_i
    float lam32[kMaxG];    // lambda'_g rounded to fp32
    double lam64[kMaxG];
};

struct FastArgs {
    const float *v;        // the unique values, times sc
    double sc, sc2, isc2;  // sc: a power of two (Prefix::scale32 = sc^2); the fp32 costs are sc2 times the binary64 ones
    const float *wf;       // multiplicities as fp32 (exact below 2^24)
    const int64_t *N;
    const double *S, *S2;  // hi [p+1] | lo [p+1]
    int64_t p, d;
    int64_t ps;            // table row stride (multiple of 64)
    float invd;            // correctly rounded 1/d
    int G, s, nJ;
    int Gc, nsplit;        // far phase: multipliers per split (Gc (s-2) <= 128 tasks), splits
    const FastParams *prm;
    float *dp32;           // tile-major fp32 copy of dp: see d32()
    uint64_t *band;        // [G][s+1][ps] tile runs per output
    int32_t *mcnt;         // [G][s+1][ps] band members
    int32_t *members;      // [G][s+1][ps][NMEM]
    uint8_t *need;         // [G][s+1][ps] output resolved exactly
    float *corner;         // [nJ(nJ-1)/2][8]: state of pair (64K+63, 64J), K < J (N, E, Ec, A, Ac, C, Cc)
    const float *costs;    // resident interval costs (tile (K, J) at J(J+1)/2 + K - tile_base), or null
    float2 *tsum;          // per tile, the summaries {min_k C, min_k Phi} of its 64 columns (the rows' padding);
                           // a value is negated where it is not the one at the tile's last k
    size_t tile_base;      // index of the first tile the costs hold: 0, or J0(J0+1)/2 for a band of blocks
    int J0, J1;            // the wavefront's column blocks [J0, J1): all of them, or one band (streamed costs)
    int build;             // the costs hold one panel's tiles, built by the wavefront itself
    int T;                 // column blocks per panel
    int workers;           // CTAs that share the far tiles
    int tcap;              // tasks per far list entry, at most (16 .. 64)
    int first_ord;         // ordinal of a far segment's first tile: 0 (higher in the test hook: shorter parts)
    float *part;           // [workers + T nsplit] segments: minima [Gc][s-2][64], then runs (seg_min, seg_runs)
    uint4 *fbits;          // far tasks: 128 bits a tile, [T nsplit][ceil(nJ/32)][32] (mask_phase)
    uint32_t *funion;      // ... and per word of 32 tiles those with any
    int *fweight;          // ... and their work
    unsigned long long *work;  // tasks evaluated in the pass
    int *tmin;             // near minima by tile group [near_groups(T)][G][s-2][64], tagged with the panel's parity
    float *tmin1;          // near minima by tile [T(T+1)/2][G][s-2][64]
    int32_t *lists;        // [s+1][2][G ps]: needed outputs of layer i (g << 24 | j); 0: <= NMEM members, 1: more
    int *list_cnt;         // [s+1][2]
    int32_t *wide;         // [G ps]: needed outputs of the layer being closed whose bands span more than
                           // kThreadTiles tiles (g << 24 | j), walked by a warp each (k_need_wide)
    int *wide_cnt;         // [s+1]
    float *mdp;            // [nJ][G][mdp_stride]: at i - 2, the min over the block's 64 columns of dp32(g, i, .)
    int mdp_stride;        // s + 1 rounded up to a multiple of 4 (16-byte rows)
    int nstage;            // stage buffers of the bound and mask phases: 2, or 1 where two do not fit shared memory
    int bound;             // the far phase starts from upper bounds of the minima (bound_phase)
    int bound_step;        // ... from every bound_step-th tile (4; 32 in unseeded searches)
    float *dlast;          // [nJ][G][mdp_stride]: at i - 2, dp32(g, i, .) at the block's last column
    int *ub;               // [T][G][s-2][64]: the bounds' float bits
    const float *seed;     // fp32 dp rows [nJ][s+1][64] of an earlier pass at a multiplier >= every
                           // multiplier of this one (upper bounds of this pass's fp32 minima), or null
    uint32_t spin_limit;   // waits on other CTAs give up after this many polls (kSpinLimit; lower in the test hook)
    int hold0;             // test hook: column block 0's minima are never written and CTA 0 stays out of the
                           // panel's barrier (their waiters time out)
    int *gbar;             // grid barrier arrivals
    int *abort_flag;
    DevStatus *st;
};

// The fp32 copy of dp is stored tile-major, [column block][g][i][64], so that the
// rows (g, i = 2..s-1) one tile of k needs are one contiguous run per multiplier.
__device__ __forceinline__ size_t d32(const FastArgs &a, int g, int i, int64_t j) {
    return (((size_t)(j >> 6) * (size_t)a.G + (size_t)g) * (size_t)(a.s + 1) + (size_t)i) * BJ + (size_t)(j & 63);
}

__device__ __forceinline__ size_t oidx(const FastArgs &a, int g, int i, int64_t j) {
    return ((size_t)g * (size_t)(a.s + 1) + (size_t)i) * (size_t)a.ps + (size_t)j;
}

// ------------------------------------------------------------ named barriers
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// BAR_BUILD .. + 5: the six 64-thread groups that build tiles; BAR_NEAR, + 1: a multiplier's eight near
// warps
enum { BAR_BUILD = 1, BAR_NEAR = 7 };
constexpr int kBuildGroups = 6;  // what shared memory stages

// Anchor of a tile: the state of pair (k, j) from double-double prefix sums.
__device__ __forceinline__ void split_f(dd x, float &hi, float &lo) {
    double t = dd_round(x);
    hi = __double2float_rn(t);
    lo = __double2float_rn(__dadd_rn(__dsub_rn(x.hi, (double)hi), x.lo));
}

__device__ void rec_anchor(const FastArgs &a, int64_t k, int64_t j, Rec &r) {
    int64_t n = a.N[j + 1] - a.N[k + 1];
    double nd = (double)n;
    dd dS = dd_sub(load_dd(a.S, a.p, j + 1), load_dd(a.S, a.p, k + 1));
    dd dS2 = dd_sub(load_dd(a.S2, a.p, j + 1), load_dd(a.S2, a.p, k + 1));
    if (a.sc2 != 1.0) {
        dS = {dS.hi * a.sc, dS.lo * a.sc};
        dS2 = {dS2.hi * a.sc2, dS2.lo * a.sc2};
    }
    double vk = (double)a.v[k], vj = (double)a.v[j];
    dd A = dd_sub(dS, two_prod(vk, nd));
    dd E = dd_sub(two_prod(vj, nd), dS);
    dd Cd = dd_sub(dd_sub(dd_mul(two_sum(vk, vj), dS), dS2), two_prod(__dmul_rn(vk, vj), nd));
    r.N = (float)n;
    split_f(E, r.E, r.Ec);
    split_f(A, r.A, r.Ac);
    split_f(Cd, r.C, r.Cc);
}

__device__ __forceinline__ size_t corner_idx(int64_t K, int64_t J) { return (size_t)J * (size_t)(J - 1) / 2 + (size_t)K; }

// Corner states (double-double, rounded to fp32 pairs) for every tile below the
// diagonal: pair (k, j) = (64K + 63, 64J), K < J.
__global__ void k_corners(FastArgs a) {
    int64_t n = (int64_t)a.nJ * (a.nJ - 1) / 2;
    int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; id < n; id += stride) {
        // invert id = J(J-1)/2 + K
        int64_t J = (int64_t)((1.0 + sqrt(1.0 + 8.0 * (double)id)) * 0.5);
        while (J * (J - 1) / 2 > id) J--;
        while ((J + 1) * J / 2 <= id) J++;
        int64_t K = id - J * (J - 1) / 2;
        Rec r;
        rec_anchor(a, K * BK + BK - 1, J * BJ, r);
        float *o = a.corner + 8 * (size_t)id;
        o[0] = r.N; o[1] = r.E; o[2] = r.Ec; o[3] = r.A; o[4] = r.Ac; o[5] = r.C; o[6] = r.Cc; o[7] = 0.f;
    }
}

// Compensated (Sum2) exclusive scan over the 64 threads jl = 0..63 of (x, c) pairs.
__device__ __forceinline__ void pair_add(float &x, float &c, float y, float yc) {
    float s = __fadd_rn(x, y);
    float bb = __fsub_rn(s, x);
    float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(y, bb));
    x = s;
    c = __fadd_rn(__fadd_rn(c, yc), e);
}

__device__ void scan64_excl(float v, float &x_out, float &c_out, float (*wsum)[2], int jl, int bar) {
    const int lane = jl & 31, wid = jl >> 5;
    float x = v, c = 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        float y = __shfl_up_sync(0xffffffffu, x, o), yc = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) pair_add(x, c, y, yc);
    }
    if (lane == 31) { wsum[wid][0] = x; wsum[wid][1] = c; }
    bar_sync(bar, NPROD);
    if (wid == 1) pair_add(x, c, wsum[0][0], wsum[0][1]);
    // exclusive: shift by one
    float xe = __shfl_up_sync(0xffffffffu, x, 1), ce = __shfl_up_sync(0xffffffffu, c, 1);
    if (lane == 0) {
        if (wid == 0) { xe = 0.f; ce = 0.f; }
        else { xe = wsum[0][0]; ce = wsum[0][1]; }
    }
    x_out = xe;
    c_out = ce;
    bar_sync(bar, NPROD);
}

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// packed fp32 pair arithmetic (sm_100+)
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
// ------------------------------------------- bulk copies (TMA engine) and mbarriers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// arrive once and raise the phase's expected transaction count by `bytes`
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait for phase `parity` of `bar`: on expiry record a timeout, raise the abort flag and return.
__device__ __forceinline__ void mbar_wait_bounded(unsigned long long *bar, uint32_t parity, DevStatus *st, int *abort_flag) {
    uint32_t spins = 0;
    while (!mbar_test(bar, parity)) {
        if (++spins > kCopySpinLimit) {
            st->timeout = 1;
            atomicExch(abort_flag, 1);
            return;
        }
        __nanosleep(32);
    }
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// global -> shared, completion counted on `bar` (bytes and both addresses multiples of 16)
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, unsigned long long *bar,
                                         uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
// shared -> global, bulk-group completion
__device__ __forceinline__ void bulk_s2g(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}
// global -> shared without a cache hint (rows every later block reads again)
__device__ __forceinline__ void bulk_g2s_nohint(void *dst, const void *src, uint32_t bytes, unsigned long long *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// generic-proxy writes to shared memory -> visible to later bulk copies
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__host__ __device__ __forceinline__ size_t cost_tile_idx(int64_t K, int64_t J) {
    return (size_t)J * (size_t)(J + 1) / 2 + (size_t)K;
}

// ------------------------------------------------------------ shared memory
// One panel: column blocks P0 .. P0 + nb - 1; its cost tiles are stored from linear index tbase.
// The far lists have nb * nsplit rows (js = split * nb + Jl) of nB words, one bit per tile.
struct Panel {
    int P0, nb, nB, tag;
    size_t tbase;
};

constexpr int NT = 32;  // tiles per word of the far lists, and per staged batch

struct __align__(16) Smem {
    float tau[kMaxS + 1];                 // FastParams::tau and lam32, read on every tile
    float lam32[kMaxG];
    uint32_t tw[8 * 16];                  // mask phase: a word of each multiplier and layer (kBoundL)
    int jstart[16 * kMaxG + 1];           // far phase: the work before each row of the list (far_plan)
    int share, first, fpos, total;        // ... the CTAs' share; this CTA's first word, its position; all work
    float gmin[NT / 8][kMaxG][16];        // mask phase: block minima of groups of eight tiles
    // far phase: the CTA's next entries (far_list) and the state of the list
    __align__(16) uint4 lbits[320];
    uint32_t lkey[320], lwhere[320];      // ... js << 14 | K; J | first multiplier << 16
    uint16_t tdiv[32 * kTaskWords];       // ... li | gl << 8 of task t
    int2 lwords[MAXCONS / 32];
    int lnext, lpos, lcount, lmore;
    __align__(16) uint32_t tinfo[4][64];  // ... entry i's tasks at i % 4: t | li << 8 | gl << 16 in row order
    __align__(16) float tlam[4][64];      // ... and their multipliers
    uint16_t okey[256];                   // ... K of a segment's tiles by ordinal (runs_add)
    int ok;                               // grid_sync's answer
    unsigned long long full[3];           // ... copies of tile buffer b
    unsigned long long smbar[2];          // copies of stage buffer sb
    unsigned long long nbar;              // copies of the near tiles
    // followed (dynamic, at kSmemHead) by one area that the phases use in turn: the far phase's tile
    // buffers (costs, then a dp32 row a task), band state and partial minima, the bound and mask phases' two stage
    // buffers and limits, the near phase's tiles and rows, or the build groups' staging
};
constexpr size_t kSmemHead = (sizeof(Smem) + 127) & ~(size_t)127;

// ------------------------------------------------------- one tile of interval costs
// Global inputs of column jl of tile (K, J), loaded by one of the 64 threads: the tile
// constants of k = 64K + jl (v_k, w_{k+1}, v_{k+1} - v_k), the column's increment
// (w_{jt+1}, v_{jt+1}, v_jt, jt = 64J + jl) and v_j, and off the diagonal the corner
// state of (K, J).
struct TileIn {
    float kv, kw, kd;
    float wn, vn, vt, vj;
    float c[7];
};
__device__ __forceinline__ void tile_load_consts(const FastArgs &a, int64_t K, int jl, TileIn &q) {
    const int64_t k = K * BK + jl;
    q.kv = k < a.p ? a.v[k] : 0.f;
    q.kw = (k + 1 < a.p) ? a.wf[k + 1] : 0.f;
    q.kd = (k + 1 < a.p) ? __fsub_rn(a.v[k + 1], a.v[k]) : 0.f;
}
__device__ __forceinline__ void tile_load(const FastArgs &a, int64_t K, int64_t J, int jl, TileIn &q) {
    const int64_t jt = J * BJ + jl;
    const bool okc = jt + 1 < a.p;
    q.wn = okc ? a.wf[jt + 1] : 0.f;
    q.vn = okc ? a.v[jt + 1] : 0.f;
    q.vt = okc ? a.v[jt] : 0.f;
    q.vj = jt < a.p ? a.v[jt] : 0.f;
#pragma unroll
    for (int r = 0; r < 7; r++) q.c[r] = 0.f;
    if (K != J) {
        const float *cp = a.corner + 8 * corner_idx(K, J);
#pragma unroll
        for (int r = 0; r < 7; r++) q.c[r] = cp[r];
    }
}

// Anchor of column jl at k = 64K + 63 (off the diagonal): the corner state of (K, J)
// advanced along j with compensated exclusive scans of non-negative increments.
// 64 threads (jl = 0..63) call it together (the scans synchronise them on barrier bar);
// vk = v at k = 64K + 63.
__device__ Rec tile_anchor(const TileIn &q, int64_t J, int jl, float vk, const FastArgs &a, float (*wsum)[2],
                           int bar) {
    const bool okc = J * BJ + jl + 1 < a.p;
    const float wn = q.wn, vn = q.vn;
    const float dj = okc ? __fsub_rn(vn, q.vt) : 0.f;
    const float *cp = q.c;
    float nx, nc, ax, ac, ex, ec, cx, cc;
    scan64_excl(wn, nx, nc, wsum, jl, bar);                               // N (exact)
    scan64_excl(okc ? __fmul_rn(wn, __fsub_rn(vn, vk)) : 0.f, ax, ac, wsum, jl, bar);  // A
    float Nj = __fadd_rn(cp[0], __fadd_rn(nx, nc));
    float Aj = __fadd_rn(__fadd_rn(cp[3], ax), __fadd_rn(cp[4], ac));
    scan64_excl(__fmul_rn(dj, Nj), ex, ec, wsum, jl, bar);              // E
    scan64_excl(__fmul_rn(dj, Aj), cx, cc, wsum, jl, bar);              // C
    Rec anchor_r;
    anchor_r.N = Nj;
    anchor_r.E = cp[1]; anchor_r.Ec = cp[2];
    pair_add(anchor_r.E, anchor_r.Ec, ex, ec);
    anchor_r.A = cp[3]; anchor_r.Ac = cp[4];
    pair_add(anchor_r.A, anchor_r.Ac, ax, ac);
    anchor_r.C = cp[5]; anchor_r.Cc = cp[6];
    pair_add(anchor_r.C, anchor_r.Cc, cx, cc);
    return anchor_r;
}

// Interval costs C[k, j] and Phi[k, j] of column j = 64J + jl for the 64 k of tile K
// (k descending) into Cr[jl][.] and Pr[jl][.]; +inf / 0 where k >= j or j >= p.
// anchor_r: the column's state at k = 64K + 63 (off the diagonal); vj = v_j.
__device__ void tile_rows(const FastArgs &a, int64_t K, int64_t J, int jl, const Rec &anchor_r, float vj,
                          const float *kv, const float *kw, const float *kd, float (*Cr)[PSTR], float (*Pr)[PSTR]) {
    const bool diag = (K == J);
    const int64_t j0 = J * BJ;
    const int64_t j = j0 + jl;
    const float d_f = (float)a.d;
        // interval costs of column j for k in the tile (descending k); the row's
        // padding slot BK receives min_k C and min_k Phi (lower bounds for tile skipping)
        float mc = CUDART_INF_F, mp = CUDART_INF_F;
        if (j < a.p) {
            Rec r;
            int kl_hi;
            if (diag) {
                r = rec_empty();
                kl_hi = (int)(j - j0) - 1;  // k = j-1 first
                // state for k = j: empty; step to k = j-1 adds t = j
                for (int kl = BK - 1; kl > kl_hi; kl--) { Cr[jl][kl] = CUDART_INF_F; Pr[jl][kl] = 0.f; }
                if (kl_hi < BK - 1) mp = 0.f;
                for (int kl = kl_hi; kl >= 0; kl--) {
                    rec_step(r, vj, kv[kl + 1], kw[kl], kd[kl]);  // kl + 1 <= 63
                    float c, ph;
                    rec_emit(r, vj, kv[kl], d_f, a.invd, c, ph);
                    Cr[jl][kl] = c; Pr[jl][kl] = ph;
                    mc = fminf(mc, c); mp = fminf(mp, ph);
                }
            } else {
                r = anchor_r;
                Rec nxt = r;
                for (int kl = BK - 1; kl >= 0; kl--) {
                    Rec cur = nxt;
                    if (kl > 0) rec_step(nxt, vj, kv[kl], kw[kl - 1], kd[kl - 1]);  // state of k - 1
                    float c, ph;
                    rec_emit(cur, vj, kv[kl], d_f, a.invd, c, ph);
                    Cr[jl][kl] = c; Pr[jl][kl] = ph;
                    mc = fminf(mc, c); mp = fminf(mp, ph);
                }
            }
        } else {
            for (int kl = 0; kl < BK; kl++) { Cr[jl][kl] = CUDART_INF_F; Pr[jl][kl] = 0.f; }
            mp = 0.f;
        }
        // The column's summary: min C and min Phi, negated where the minimum is not the value at
        // the tile's last k (then dp(., k) + C + lambda' Phi at that k is not the summary's own).
        Cr[jl][BK] = mc == Cr[jl][BK - 1] ? mc : __int_as_float(__float_as_int(mc) | (int)0x80000000);
        Pr[jl][BK] = mp == Pr[jl][BK - 1] ? mp : __int_as_float(__float_as_int(mp) | (int)0x80000000);
}

// Interval-cost tiles t0, t0 + stride, ... below t1 (linear index J(J+1)/2 + K), each computed
// once (tile_anchor, tile_rows), staged in shared memory and written out by a bulk copy to
// costs / tsum at t - tbase.  Called by 64 threads (jl = 0..63, named barrier bar).  A tile's
// global inputs are loaded while the previous tile's rows are computed, and the wait for the
// previous bulk store to have read the staging rows comes only just before they are overwritten.
struct __align__(16) BuildSmem {
    float C[BJ][PSTR];
    float Phi[BJ][PSTR];
    float kv[BK], kw[BK], kd[BK];
    float wsum[2][2];
};

__device__ __forceinline__ void build_tiles(const FastArgs &a, BuildSmem &S, int jl, int bar, int64_t t0,
                                            int64_t stride, int64_t t1, int64_t tbase) {
    int64_t t = t0;
    if (t >= t1) return;
    // invert t = J(J+1)/2 + K, K <= J
    int64_t J = (int64_t)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while (J * (J + 1) / 2 > t) J--;
    while ((J + 1) * (J + 2) / 2 <= t) J++;
    int64_t K = t - J * (J + 1) / 2;
    TileIn cur;
    tile_load_consts(a, K, jl, cur);
    tile_load(a, K, J, jl, cur);
    for (;;) {
        S.kv[jl] = cur.kv; S.kw[jl] = cur.kw; S.kd[jl] = cur.kd;
        bar_sync(bar, NPROD);
        const Rec anchor_r = K == J ? rec_empty() : tile_anchor(cur, J, jl, S.kv[BK - 1], a, S.wsum, bar);
        // the next tile: t + stride, walking (J, K) along the rows
        const int64_t tn = t + stride;
        int64_t Jn = J, Kn = K + stride;
        while (Kn > Jn) { Kn -= Jn + 1; Jn++; }
        TileIn nxt;
        if (tn < t1) {
            tile_load_consts(a, Kn, jl, nxt);
            tile_load(a, Kn, Jn, jl, nxt);
        }
        if (jl == 0) bulk_wait_read_all();  // the previous tile's bulk store has read the rows
        bar_sync(bar, NPROD);
        tile_rows(a, K, J, jl, anchor_r, cur.vj, S.kv, S.kw, S.kd, S.C, S.Phi);
        a.tsum[(size_t)(t - tbase) * BJ + jl] = make_float2(S.C[jl][BK], S.Phi[jl][BK]);  // this thread's own row
        fence_proxy_async_smem();
        bar_sync(bar, NPROD);
        if (jl == 0) {
            float *dst = const_cast<float *>(a.costs) + (size_t)(t - tbase) * kCostTileFloats;
            bulk_s2g(dst, &S.C[0][0], kCostHalfBytes);
            bulk_s2g(dst + kCostHalfFloats, &S.Phi[0][0], kCostHalfBytes);
            bulk_commit();
        }
        if (tn >= t1) break;
        t = tn; J = Jn; K = Kn;
        cur = nxt;
    }
    if (jl == 0) bulk_wait_all();
}

static __device__ __noinline__ void build_panel(const FastArgs &a, BuildSmem &S, int jl, int bar, int64_t t0,
                                                int64_t stride, int64_t t1, int64_t tbase) {
    build_tiles(a, S, jl, bar, t0, stride, t1, tbase);  // the wavefront's: registers of its own
}

// The tiles of column blocks [J0, J1): indices J0(J0+1)/2 .. J1(J1+1)/2 - 1, stored from tile_base.
__global__ void __launch_bounds__(NPROD) k_build_costs(const __grid_constant__ FastArgs a) {
    __shared__ BuildSmem S;
    build_tiles(a, S, threadIdx.x, BAR_BUILD, (int64_t)a.tile_base + blockIdx.x, gridDim.x,
                (int64_t)a.J1 * (a.J1 + 1) / 2, (int64_t)a.tile_base);
}

// ------------------------------------------------------------ panels
// The column blocks go in panels of a.T (15 on this GPU) consecutive blocks [P0, P0 + nb), one
// after the other.  Within a panel, grid barriers between the steps:
//  1. bound_phase: upper bounds of the minima over the far tiles (K < P0, whose dp rows are all
//     final) from one candidate of every fourth tile;
//  2. mask_phase: the far tasks -- (tile, multiplier, layer) -- that may matter, by the skip test
//     against the bounds;
//  3. far_phase: the tiles with tasks in one list, an equal share of the work for each CTA; a CTA's
//     results for a column block -- a segment -- go to the outputs' minima and, with their band
//     runs, to a slot;
//  4. near_phase: the panel's own triangle of tiles, layer by layer.  A CTA takes up to four tiles
//     (K, J) of one J and two multipliers, two warps one of each, with the tile's costs
//     C + lambda' Phi in registers (a lane: one column) for all layers.  For layer i a warp gathers
//     row i-1 of its block K -- the far minimum and the (at most four) groups' minima above it --
//     and the CTA writes its group's minima of layer i.  A written minimum carries the panel's
//     parity in its sign bit (values are >= +0), so the value is its own flag: a reader polls
//     the values themselves (bounded), and no fence or counter stands between two layers;
//  5. fold_panel: every output's band from the segments' runs and the near minima.
// What bounds it: a wavefront of whole column blocks made the chain of blocks (one block's last
// tile and diagonal, every layer, 22 000 cycles at s = 16) the critical path and left the SMs
// unevenly loaded; here 15 blocks cost a few barriers and s - 2 gather/compute steps, and the
// far tiles are shared evenly.  A pass of 8 multipliers (mean over a budgeted search, resident
// costs): 22.5 ms instead of 46.3 at d = 2^17, s = 16; 1.47 instead of 2.93 at d = 16384, s = 16;
// 12.9 instead of 47.7 at d = 50001, s = 32; building its own costs, 2.4 instead of 8.4 at
// d = 12289, s = 16.  Of the 22.5 ms 11.0 are far tiles, 2.4 uneven shares, 2.8 masks, 1.4 bounds, 2.4
// the near phases, 0.8 the fold and 1.7 barriers and the rest.  Far tiles are bound by the latency of one tile's
// chain -- copies, costs into registers, a batch of tasks, a barrier, the fold: about 3000 cycles
// with eight tasks, at most 13 candidates per cycle and SM where the adds and mins alone would
// reach 53 -- so a tile costs as much as about 6 of its tasks on top of them (kTileCost).

// Grid barrier `epoch` (1, 2, ...): bounded; false when it gave up or another CTA aborted.  All
// CTAs are resident (cooperative launch).  Orders generic and bulk-copy accesses on both sides.
__device__ __forceinline__ bool grid_sync(const FastArgs &a, Smem &S, int epoch, bool arrive = true) {
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        const int target = epoch * (int)gridDim.x;
        if (arrive) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.gbar) : "memory");
        uint32_t spins = 0;
        int ok = 1;
        while (ld_acquire(a.gbar) < target) {
            if ((++spins & 63u) == 0u) {
                if (*(volatile int *)a.abort_flag) { ok = 0; break; }
                if (spins > a.spin_limit) {
                    a.st->timeout = 1;
                    atomicExch(a.abort_flag, 1);
                    ok = 0;
                    break;
                }
            }
            __nanosleep(20);
        }
        S.ok = ok;
    }
    __syncthreads();
    asm volatile("fence.proxy.async;" ::: "memory");
    return S.ok != 0;
}

// Bound and mask phases: warp 0 stages up to NT consecutive far tiles of block J -- their column
// summaries and the tiles' rows of `src` (a.dlast or a.mdp, all G multipliers) -- with two bulk copies.
__host__ __device__ __forceinline__ size_t stage_floats(int G, int mdp_stride) {
    return (size_t)NT * BJ * 2 + (size_t)NT * G * mdp_stride;
}
// Stage number ns: its buffer, and the parity of its barrier's phase.
__device__ __forceinline__ int stage_buf(const FastArgs &a, uint32_t ns) { return a.nstage == 2 ? (int)(ns & 1u) : 0; }
__device__ __forceinline__ uint32_t stage_parity(const FastArgs &a, uint32_t ns) { return (a.nstage == 2 ? ns >> 1 : ns) & 1u; }
__device__ __forceinline__ void stage_tiles(const FastArgs &a, Smem &S, float *stg, int sb, int K0, int n, int J,
                                            size_t tbase, const float *src, uint64_t policy) {
    const uint32_t tb = (uint32_t)((size_t)n * BJ * sizeof(float2));
    const uint32_t mb = (uint32_t)((size_t)n * a.G * a.mdp_stride * sizeof(float));
    mbar_expect_tx(&S.smbar[sb], tb + mb);
    bulk_g2s(stg, a.tsum + (cost_tile_idx(K0, J) - tbase) * BJ, tb, &S.smbar[sb], policy);
    bulk_g2s_nohint(stg + (size_t)NT * BJ * 2, src + (size_t)K0 * a.G * a.mdp_stride, mb, &S.smbar[sb]);
}

constexpr int kNoBound = 0x7F7F7F7F;  // bits above every finite fp32 cost that occurs; a byte pattern (memset)
__device__ __forceinline__ int *ub_at(const FastArgs &a, int Jl, int g) {
    return a.ub + ((size_t)Jl * a.G + g) * (size_t)(a.s - 2) * BJ;
}

// Upper bounds of the panel's far minima: for every output the least candidate over the last k
// of every fourth far tile (a.bound_step), dp(i-1, 64K+63) + C + lambda' Phi with C and Phi from the tile's
// summary (where the summary is that k's, which it nearly always is) -- a candidate's own fp32 value, so never
// below the minimum, and within the change of the candidates over a few tiles of it.  Tiles are then
// skipped as if the minimum were known (far_start), whatever the order of the walk.  One candidate of
// 256 is evaluated for it; a budgeted search at d = 2^17, s = 16 then runs 5 % of the (tile, multiplier, layer)
// tasks (mask_phase).
// CTAs split the panel's (column block, tile range) pairs evenly; a thread owns one column of one
// multiplier, kBoundL layers at a time.
constexpr int kBoundL = 16;
static __device__ __noinline__ void bound_phase(const FastArgs &a, Smem &S, float *stage, const Panel &pn,
                                                uint64_t policy, uint32_t &ns) {
    const int L = a.s - 2, ct = threadIdx.x, jl = ct & (BJ - 1), gq = ct / BJ;
    const size_t sfl = stage_floats(a.G, a.mdp_stride);
    const int parts = max(1, (int)gridDim.x / pn.nb);
    const int Jl = (int)blockIdx.x % pn.nb, part = (int)blockIdx.x / pn.nb;
    if (part >= parts) return;
    const int Ka = (int)((int64_t)pn.P0 * part / parts), Kb = (int)((int64_t)pn.P0 * (part + 1) / parts);
    if (Ka >= Kb) return;
    const int J = pn.P0 + Jl, g = min(gq, a.G - 1);
    const float lam = S.lam32[g];
    for (int l0 = 0; l0 < L; l0 += kBoundL) {
        int m[kBoundL];
#pragma unroll
        for (int l = 0; l < kBoundL; l++) m[l] = 0x7f800000;
        auto stage_from = [&](int K) {
            const int sb = stage_buf(a, ns);
            stage_tiles(a, S, stage + sb * sfl, sb, K, min(NT, Kb - K), J, pn.tbase, a.dlast, policy);
        };
        if (ct == 0) stage_from(Ka);
        for (int K0 = Ka; K0 < Kb; K0 += NT) {
            const int n = min(NT, Kb - K0), sb = stage_buf(a, ns);
            const float *stg = stage + sb * sfl;
            const uint32_t ph = stage_parity(a, ns);
            ns++;
            const bool more = K0 + NT < Kb && ct == 0;
            if (more && a.nstage == 2) stage_from(K0 + NT);
            mbar_wait_bounded(&S.smbar[sb], ph, a.st, a.abort_flag);
            const float2 *ts = reinterpret_cast<const float2 *>(stg) + jl;
            const float *d = stg + (size_t)NT * BJ * 2 + l0 + (size_t)g * a.mdp_stride;
            const int rs = a.G * a.mdp_stride, step = a.bound_step;
#pragma unroll 2
            for (int r = (step - K0 % step) % step; r < n; r += step) {
                const float2 v = ts[r * BJ];
                const bool last = (__float_as_int(v.x) | __float_as_int(v.y)) >= 0;
                const float w = last ? __fmaf_rn(lam, v.y, v.x) : CUDART_INF_F;
#pragma unroll
                for (int l = 0; l < kBoundL; l += 4)
                    if (l0 + l < L) {  // the rows are padded to a multiple of four
                        const float4 x = *reinterpret_cast<const float4 *>(d + r * rs + l);
                        m[l] = min(m[l], __float_as_int(__fadd_rn(x.x, w)));
                        m[l + 1] = min(m[l + 1], __float_as_int(__fadd_rn(x.y, w)));
                        m[l + 2] = min(m[l + 2], __float_as_int(__fadd_rn(x.z, w)));
                        m[l + 3] = min(m[l + 3], __float_as_int(__fadd_rn(x.w, w)));
                    }
            }
            __syncthreads();  // the stage buffer is free
            if (more && a.nstage != 2) stage_from(K0 + NT);
        }
#pragma unroll
        for (int l = 0; l < kBoundL; l++)
            if (l0 + l < L && gq < a.G && m[l] < kNoBound)
                atomicMin(ub_at(a, Jl, gq) + (size_t)(l0 + l) * BJ + jl, m[l]);
    }
}

// The far phase starts each output's running minimum from +inf, lowered by an earlier pass's minimum
// (a.seed) and the panel's bound.  Every fp32 candidate is monotone in lambda' (C and Phi are >= 0 and
// the roundings are monotone), so by induction over the layers an earlier pass's fp32 minimum at a
// multiplier >= this one's bounds this pass's minimum m from above, as a candidate's own value does.
// Starting at any such bound changes no result: the tile holding m is never skipped (its lower bound is
// <= m <= the limit), so the final minimum is m itself; a tile the tighter limit skips has every
// candidate above m (1 + tau), outside the band; and the walk keeps the band a superset of the tiles with
// a candidate within m (1 + tau) from any starting bb >= m (a reset drops only tiles whose candidates all
// lie above the band).  A walk that records no tile adds none to the band.  Only the skip tests
// see the start.
__device__ __forceinline__ float far_bound(int w) { return w < kNoBound ? __int_as_float(w) : CUDART_INF_F; }
// ... of the four outputs o .. o + 3 of a split and column block J: o = t * 64 + column, t = gl * L + li; u: the
// split's bounds (ub_at).
__device__ __forceinline__ float4 far_start(const FastArgs &a, const int *u, int J, int o) {
    float4 v = make_float4(CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, CUDART_INF_F);
    if (a.bound) {
        const int4 w = __ldcg(reinterpret_cast<const int4 *>(u + o));
        v = make_float4(far_bound(w.x), far_bound(w.y), far_bound(w.z), far_bound(w.w));
    }
    if (a.seed) {  // (columns past the last value hold +inf)
        const float4 x = __ldg(reinterpret_cast<const float4 *>(
            a.seed + ((size_t)J * (size_t)(a.s + 1) + 3 + (o / BJ) % (a.s - 2)) * BJ + (o & (BJ - 1))));
        v = make_float4(fminf(v.x, x.x), fminf(v.y, x.y), fminf(v.z, x.z), fminf(v.w, x.w));
    }
    return v;
}

// The far tasks: task t = gl * L + li of a multiplier split (multiplier split * Gc + gl, layer 3 + li) on a
// tile, needed when some column may take a candidate from the tile.  The test is exact skipping: every
// candidate of the tile for an output is >= lb = fl(min dp(i-1, .) + fl(fma(lam, min Phi, min C))) (rounding
// is monotone); when lb exceeds the output's band limit bb + bb tau, the tile changes neither its
// minimum nor its band.  For row js = split * nb + Jl, a.fbits has 128 task bits a tile, and for each word
// of 32 tiles a.funion says which have any and a.fweight the word's work: the tasks, and kTileCost a tile.
// A tile that is copied in has 14 of its 112 tasks needed at d = 2^17, s = 16 (mean of a search), so
// tasks, not whole tiles, are the unit of work.
// CTAs split the (column block, word range) pairs as in bound_phase; a thread tests one column of one
// multiplier, kBoundL layers at a time.
constexpr int kTileCost = 6;  // a listed tile's fixed cost (its copies, its costs into registers) in tasks (a pass at d = 2^17, s = 16: 22.5 ms
                               // with 6, 23.9 with 3, 23.0 with 9)
static __device__ __noinline__ void mask_phase(const FastArgs &a, Smem &S, float *stage, const Panel &pn,
                                               uint64_t policy, uint32_t &ns) {
    const int L = a.s - 2, ct = threadIdx.x, lane = ct & 31, wid = ct >> 5, jl = ct & (BJ - 1), gq = ct / BJ;
    const size_t sfl = stage_floats(a.G, a.mdp_stride);
    const int parts = max(1, (int)gridDim.x / pn.nb);
    const int Jl = (int)blockIdx.x % pn.nb, part = (int)blockIdx.x / pn.nb, J = pn.P0 + Jl;
    if (part >= parts) return;
    const int ba = pn.nB * part / parts, bz = pn.nB * (part + 1) / parts;
    if (ba >= bz) return;
    auto stage_word = [&](int b) {
        const int sb = stage_buf(a, ns);
        stage_tiles(a, S, stage + sb * sfl, sb, b * NT, min(NT, pn.P0 - b * NT), J, pn.tbase, a.mdp, policy);
    };
    for (int split = 0; split < a.nsplit; split++) {
        if (ct == 0) stage_word(ba);
        // the outputs' band limits, into shared memory: one coalesced read, whatever the layers' order
        float *slim = stage + a.nstage * sfl;  // [Gc][L][64]
        const int gs = split * a.Gc, ngv = min(a.Gc, a.G - gs);
        const int *u = ub_at(a, Jl, gs);
        for (int o = 4 * ct; o < ngv * L * BJ; o += 4 * MAXCONS) {
            const float4 v = far_start(a, u, J, o);
            const float tau = S.tau[3 + (o / BJ) % L];
            *reinterpret_cast<float4 *>(slim + o) =
                make_float4(__fadd_rn(v.x, __fmul_rn(v.x, tau)), __fadd_rn(v.y, __fmul_rn(v.y, tau)),
                            __fadd_rn(v.z, __fmul_rn(v.z, tau)), __fadd_rn(v.w, __fmul_rn(v.w, tau)));
        }
        const bool own = gq < ngv;
        const int g = gs + (own ? gq : 0);
        const float lam = S.lam32[g];
        for (int b = ba; b < bz; b++) {
            const int n = min(NT, pn.P0 - b * NT), sb = stage_buf(a, ns);
            const float *stg = stage + sb * sfl, *md = stg + (size_t)NT * BJ * 2;
            const uint32_t ph = stage_parity(a, ns);
            const int rs = a.G * a.mdp_stride;
            ns++;
            const bool more = b + 1 < bz && ct == 0;
            if (more && a.nstage == 2) stage_word(b + 1);
            if (ct < 32 * kTaskWords) S.tw[ct] = 0u;
            mbar_wait_bounded(&S.smbar[sb], ph, a.st, a.abort_flag);
            for (int l0 = 0; l0 < L; l0 += kBoundL) {
                // block minima of groups of eight tiles
                for (int q = ct; q < NT / 8 * kMaxG * kBoundL; q += MAXCONS) {
                    const int grp = q / (kMaxG * kBoundL), gg = (q / kBoundL) % kMaxG, l = q % kBoundL;
                    float m = CUDART_INF_F;
                    if (gg < a.G && l0 + l < L)
#pragma unroll
                        for (int x = 0; x < 8; x++)
                            if (8 * grp + x < n) m = fminf(m, md[(8 * grp + x) * rs + gg * a.mdp_stride + l0 + l]);
                    S.gmin[grp][gg][l] = m;
                }
                __syncthreads();  // tw is clear, gmin and slim complete
                float lim[kBoundL];
                uint32_t mine[kBoundL];
#pragma unroll
                for (int l = 0; l < kBoundL; l++) {
                    mine[l] = 0u;
                    lim[l] = (own && l0 + l < L) ? slim[((g - gs) * L + l0 + l) * BJ + jl] : -1.f;
                }
                const float2 *ts = reinterpret_cast<const float2 *>(stg) + jl;
                for (int grp = 0; 8 * grp < n; grp++) {
                    // a group of eight tiles at a time: the group's least block minimum and summaries bound
                    // every tile of it, and only a layer that some lane may need there is tested tile by tile
                    float lb[8], cx = CUDART_INF_F, cy = CUDART_INF_F;
#pragma unroll
                    for (int x = 0; x < 8; x++) {
                        const float2 v = ts[(8 * grp + x) * BJ];
                        const bool in = 8 * grp + x < n;  // (rows past n hold anything; their bits are dropped)
                        const float c = fabsf(v.x), f = fabsf(v.y);
                        lb[x] = __fmaf_rn(lam, f, c);
                        cx = in ? fminf(cx, c) : cx;
                        cy = in ? fminf(cy, f) : cy;
                    }
                    const uint32_t valid = n - 8 * grp >= 8 ? 0xffu : (1u << (n - 8 * grp)) - 1u;
                    const float gb = __fmaf_rn(lam, cy, cx);
                    const float *gm = S.gmin[grp][g];
                    const float *d = md + (size_t)(8 * grp) * rs + (size_t)g * a.mdp_stride + l0;
#pragma unroll
                    for (int l = 0; l < kBoundL; l++)
                        if (__any_sync(0xffffffffu, __fadd_rn(gm[l], gb) <= lim[l])) {
                            uint32_t m = 0u;
#pragma unroll
                            for (int x = 0; x < 8; x++) m |= (__fadd_rn(d[x * rs + l], lb[x]) <= lim[l] ? 1u : 0u) << x;
                            mine[l] |= (m & valid) << (8 * grp);
                        }
                }
                // the union over the 64 columns: two warps a multiplier
#pragma unroll
                for (int l = 0; l < kBoundL; l++) {
                    const uint32_t m = __reduce_or_sync(0xffffffffu, mine[l]);
                    if (lane == 0 && m) atomicOr(&S.tw[(g - gs) * L + l0 + l], m);
                }
                __syncthreads();  // this part of tw is complete; gmin is free
            }
            // a warp turns two tiles' bits round; word totals by the first warp
            const size_t w = (size_t)(split * pn.nb + Jl) * pn.nB + b;
            uint32_t word[kTaskWords];
#pragma unroll
            for (int x = 0; x < kTaskWords; x++) word[x] = S.tw[lane + 32 * x];
#pragma unroll
            for (int y = 0; y < NT / (MAXCONS / 32); y++) {
                const int r = NT / (MAXCONS / 32) * wid + y;
                uint32_t bits[kTaskWords];
#pragma unroll
                for (int x = 0; x < kTaskWords; x++) bits[x] = __ballot_sync(0xffffffffu, (word[x] >> r) & 1u);
                if (lane == 0) __stcg(a.fbits + w * NT + r, make_uint4(bits[0], bits[1], bits[2], bits[3]));
            }
            if (wid == 0) {
                uint32_t any = 0u;
                int work = 0;
#pragma unroll
                for (int x = 0; x < kTaskWords; x++) { any |= word[x]; work += __popc(word[x]); }
                any = __reduce_or_sync(0xffffffffu, any);
                work = __reduce_add_sync(0xffffffffu, work);
                if (lane == 0) {
                    a.funion[w] = any;
                    a.fweight[w] = work + kTileCost * __popc(any);
                }
            }
            __syncthreads();  // tw and, of one, the stage buffer are free
            if (more && a.nstage != 2) stage_word(b + 1);
        }
    }
}

// The position (in work) where each row of the list starts (S.jstart), the CTAs' share (S.share),
// this CTA's first word (S.first) and the position where it starts (S.fpos).  Every CTA computes the same.
__device__ __forceinline__ void far_plan(const FastArgs &a, Smem &S, const Panel &pn) {
    const int ct = threadIdx.x, lane = ct & 31, wid = ct >> 5, nj = pn.nb * a.nsplit;
    for (int js = wid; js < nj; js += MAXCONS / 32) {
        int n = 0;
        for (int b = lane; b < pn.nB; b += 32) n += __ldcg(a.fweight + (size_t)js * pn.nB + b);
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) S.jstart[js + 1] = n;
    }
    __syncthreads();
    if (wid == 0) {
        int run = 0;
        for (int j0 = 0; j0 < nj; j0 += 32) {
            int v = j0 + lane < nj ? S.jstart[j0 + lane + 1] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += x;
            }
            if (j0 + lane < nj) S.jstart[j0 + lane + 1] = run + v;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) S.jstart[0] = 0;
        const int share = max(1, (run + a.workers - 1) / a.workers);
        const int pos0 = (int)blockIdx.x * share;
        __syncwarp();
        int first = -1, fpos = 0;
        if ((int)blockIdx.x < a.workers && pos0 < run) {
            // the row that holds pos0, then its word
            int js = 0;
            for (int j0 = 0; j0 < nj; j0 += 32) {
                const unsigned in = __ballot_sync(0xffffffffu, j0 + lane < nj && S.jstart[j0 + lane] <= pos0 &&
                                                                   S.jstart[j0 + lane + 1] > pos0);
                if (in) js = j0 + __ffs(in) - 1;
            }
            int before = S.jstart[js];
            for (int b0 = 0; b0 < pn.nB && first < 0; b0 += 32) {
                const int b = b0 + lane;
                int v = b < pn.nB ? (int)__ldcg(a.fweight + (size_t)js * pn.nB + b) : 0;
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += x;
                }
                const unsigned past = __ballot_sync(0xffffffffu, before + v > pos0);
                if (past) {
                    const int l = __ffs(past) - 1;
                    first = js * pn.nB + b0 + l;
                    fpos = before + (l ? __shfl_sync(0xffffffffu, v, l - 1) : 0);
                }
                before += __shfl_sync(0xffffffffu, v, 31);
            }
        }
        if (lane == 0) {
            S.share = share;
            S.first = first;
            S.fpos = fpos;
            S.total = run;
        }
    }
    __syncthreads();
}

// A segment's slot: worker c's results for row js.  (c, js) pairs with work form a monotone path,
// so c + js names each once.
__device__ __forceinline__ float *seg_min(const FastArgs &a, int c, int js) {
    return a.part + (size_t)(c + js) * a.Gc * (a.s - 2) * BJ * 3;
}
__device__ __forceinline__ uint2 *seg_runs(const FastArgs &a, float *seg) {
    return reinterpret_cast<uint2 *>(seg + (size_t)a.Gc * (a.s - 2) * BJ);
}

// The far phase of one panel: this CTA's share of the list, the tiles whose position lies in
// [share c, share (c + 1)), in entries of at most a.tcap tasks.  Sixteen warps take 8 of the tile's 64 k and
// 32 of its columns each, the costs in registers (a lane: one column), and go through the entry's tasks
// eight at a time: C + lambda' Phi, the task's dp row (one address a warp: a single
// shared-memory access), the least of 8 candidates into a slot of the column's eight partial minima.
// After one barrier a pair of warps takes each of the eight tasks, and a lane folds its column's minimum
// into the band state (shared memory) while the next eight tasks start.  So a tile's costs are read
// once and the warps are always even.  Shared-memory traffic is what such a loop has to save: with lanes on
// eight k groups of four columns it took 330 cycles a task, with atomics in place of the slots 280, and
// a warp of one multiplier with 28 outputs a lane in registers took 10 000 cycles a tile whatever it
// needed of it.
constexpr int kFarBufs = 3;
constexpr int kBatch = 8;      // tasks between two barriers
constexpr int kFarList = 320;  // list entries held
struct Pipe {
    uint32_t n, ns, nnear;  // far entries, stage fills and near tiles so far
    uint32_t run, fetched;  // tasks evaluated; tiles copied in
};
__device__ __forceinline__ float *far_buf(const FastArgs &a, float *big, int b) {
    return big + (size_t)b * (kCostTileFloats + (size_t)a.tcap * BK);
}

// The first task of a tile of n (its position: its work before it, then kTileCost, then its tasks) behind a
// share's border at `x` from the tile's position.  A border divides a tile's tasks, in eights, where both sides
// keep 16 or more, as a tile of 112 tasks is a whole share of a small panel (d = 16384: 1.69 ms a pass with
// whole tiles, 1.55 now); else they go to the later share.
__device__ __forceinline__ int share_cut(int x, int n) {
    x -= kTileCost;
    if (x >= n) return n;
    if (x < 16) return 0;
    return n - x < 16 ? n : x & ~7;
}

// The next entries of the share, from word S.lnext (whose position is S.lpos) on: up to 16 words, a warp
// each, as many as the list holds.  An entry: js << 14 | K, and its tasks as 128 bits.  S.lcount: entries;
// S.lmore: the share goes on.  All threads.
__device__ __forceinline__ void far_list(const FastArgs &a, Smem &S, const Panel &pn) {
    constexpr int kW = MAXCONS / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwords = pn.nb * a.nsplit * pn.nB;
    const int pos0 = (int)blockIdx.x * S.share, end = min(pos0 + S.share, S.total);
    const int e0 = S.lnext, e = e0 + wid;
    // the words' positions
    const int fw = lane < kW && e0 + lane < nwords ? __ldcg(a.fweight + e0 + lane) : 0;
    uint32_t u = e < nwords ? __ldcg(a.funion + e) : 0u;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if ((u >> lane) & 1u) v = __ldcg(a.fbits + (size_t)e * NT + lane);
    int before = fw;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += x;
    }
    const int after = S.lpos + __shfl_sync(0xffffffffu, before, kW - 1);  // position after the sixteen words
    const int wpos = S.lpos + __shfl_sync(0xffffffffu, before - fw, wid);
    // the word's tiles: position, in the share or not, entries
    const int n = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    const int weight = n ? n + kTileCost : 0;
    int pos = weight;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, pos, o);
        if (lane >= o) pos += x;
    }
    pos += wpos - weight;
    const int lo = share_cut(pos0 - pos, n), cnt = share_cut(end - pos, n) - lo;  // the share's tasks of the tile
    const bool mine = cnt > 0;
    const int parts = mine ? (cnt + a.tcap - 1) / a.tcap : 0;
    int at = parts;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += x;
    }
    const int total = __shfl_sync(0xffffffffu, at, 31);
    if (lane == 0) S.lwords[wid] = make_int2(total, wpos);
    __syncthreads();
    int off = 0, used = 0, all = 0;  // entries of the words before; words taken and their entries
    for (int w = 0; w < kW; w++) {
        const int c = S.lwords[w].x;
        if (w < wid) off += c;
        if (used == w && all + c <= kFarList) {
            used++;
            all += c;
        }
    }
    if (wid < used && mine) {
        const int js = e / pn.nB, K = (e - js * pn.nB) * NT + lane, split = js / pn.nb;
        uint32_t bits[kTaskWords] = {v.x, v.y, v.z, v.w};
        int skip = lo, left = cnt;
#pragma unroll
        for (int x = 0; x < kTaskWords; x++)
            for (; skip > 0 && bits[x]; skip--) bits[x] &= bits[x] - 1u;
        for (int p = 0, i = off + at - parts; p < parts; p++, i++) {  // at most tcap tasks each, lowest first
            const int cap = min(a.tcap, left);
            left -= cap;
            uint32_t out[kTaskWords];
            int m = 0;
#pragma unroll
            for (int x = 0; x < kTaskWords; x++) {
                uint32_t take = bits[x];
                while (m + __popc(take) > cap) take &= ~(1u << (31 - __clz(take)));
                m += __popc(take);
                out[x] = take;
                bits[x] &= ~take;
            }
            S.lkey[i] = (uint32_t)js << 14 | (uint32_t)K;
            S.lwhere[i] = (uint32_t)(pn.P0 + js - split * pn.nb) | (uint32_t)(split * a.Gc) << 16;
            S.lbits[i] = make_uint4(out[0], out[1], out[2], out[3]);
        }
    }
    const int2 cut = used < kW ? S.lwords[used] : make_int2(0, 0);
    __syncthreads();  // the list is complete, every thread has read lnext and lpos
    if (threadIdx.x == 0) {
        S.lcount = all;
        S.lnext = e0 + used;
        S.lpos = used < kW ? cut.y : after;
        S.lmore = e0 + used < nwords && (used < kW ? cut.y : after) < end ? 1 : 0;
    }
    __syncthreads();
}

// Copies of list entry i into buffer b, and its tasks in row order at slot `slot`: t | li << 8 | gl << 16.
// Five warps share it (role 0: the costs; 1 + x: the rows of the tasks in word x), as a warp that issued it all
// came 1000 cycles late to the next barrier.  The readers look at the slot after the buffer's phase, which takes
// one arrival of each.
__device__ __forceinline__ void far_issue(const FastArgs &a, Smem &S, float *big, const Panel &pn, int i, int slot, int b,
                                          int role, uint64_t policy) {
    const int lane = threadIdx.x & 31;
    const uint4 v = S.lbits[i];
    const uint32_t where = S.lwhere[i], bits[kTaskWords] = {v.x, v.y, v.z, v.w};
    const int K = (int)(S.lkey[i] & 0x3FFFu), J = (int)(where & 0xFFFFu), gs = (int)(where >> 16);
    float *buf = far_buf(a, big, b);
    if (role == 0) {
        if (lane == 0) {
            const int n = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            mbar_expect_tx(&S.full[b], 2 * kCostHalfBytes + (uint32_t)(n * BK * sizeof(float)));
            bulk_g2s(buf, a.costs + (cost_tile_idx(K, J) - pn.tbase) * kCostTileFloats, 2 * kCostHalfBytes, &S.full[b],
                     policy);
        }
        return;
    }
    int row = 0;
    uint32_t mine = 0u;
#pragma unroll
    for (int x = 0; x < kTaskWords; x++) {
        if (x < role - 1) row += __popc(bits[x]);
        if (x == role - 1) mine = bits[x];
    }
    if ((mine >> lane) & 1u) {
        const int t = lane + 32 * (role - 1);
        row += __popc(mine & ((1u << lane) - 1u));
        const uint32_t d = S.tdiv[t];  // li | gl << 8
        S.tinfo[slot][row] = (uint32_t)t | d << 8;
        S.tlam[slot][row] = S.lam32[gs + (int)(d >> 8)];
        bulk_g2s_nohint(buf + kCostTileFloats + row * BK,
                        a.dp32 + d32(a, gs + (int)(d >> 8), 2 + (int)(d & 0xFFu), (int64_t)K * BK),
                        (uint32_t)(BK * sizeof(float)), &S.full[b]);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.full[b]);
}

// Band runs while a segment is walked, in four bytes: first and last of run 1, then of run 2, as
// ordinals of the segment's tiles (at most 254, then the segment is stored and goes on in a next
// part); run 2 absent: 0 (its ordinals are >= 1); no tile yet: kNoRuns.  cont: this tile's K follows the
// K of the tile before.
constexpr uint32_t kNoRuns = 0xFFu;
constexpr int kLastOrd = 254;
// Runs r appended to the band word (w1, w2), in increasing K, as runs_add appends tiles.
__device__ __forceinline__ void band_append(uint32_t &w1, uint32_t &w2, bool &any, uint32_t f, uint32_t l) {
    if (!any) { w1 = (f << 16) | l; any = true; }
    else if (!w2 && (w1 & 0xFFFFu) + 1u == f) w1 = (w1 & 0xFFFF0000u) | l;
    else if (!w2) w2 = (f << 16) | l;
    else w2 = (w2 & 0xFFFF0000u) | l;
}
__device__ __forceinline__ uint32_t runs_add(uint32_t w, bool rst, uint32_t o, bool cont) {
    if (rst || w == kNoRuns) return o | o << 8;
    const bool has2 = (w >> 24) != 0u;
    if (!has2 && cont && ((w >> 8) & 0xFFu) + 1u == o) return (w & 0xFFu) | o << 8;
    return has2 ? (w & 0x00FFFFFFu) | o << 24 : (w & 0xFFFFu) | o << 16 | o << 24;
}

__device__ __forceinline__ void far_phase(const FastArgs &a, Smem &S, float *big, const Panel &pn, uint64_t policy,
                                          Pipe &pp) {
    const int L = a.s - 2, nt = a.Gc * L, ct = threadIdx.x, lane = ct & 31, wid = ct >> 5;
    const int slice = wid & 7, col = lane + 32 * (wid >> 3);
    if (S.first < 0) return;
    float *sbest = far_buf(a, big, kFarBufs);
    uint32_t *sruns = reinterpret_cast<uint32_t *>(sbest + (size_t)nt * BJ);
    int *part = reinterpret_cast<int *>(sruns + (size_t)nt * BJ);  // [2][kBatch][8][64]
    int js = -1, ord = 0, lastK = -2;
    bool cont = false, next = false;  // next: not the segment's first part
    // all threads: the segment's minima into the outputs, minima and runs to its slot, behind those of its parts before
    auto flush = [&]() {
        const int split = js / pn.nb, real = min(a.Gc, a.G - split * a.Gc) * L * BJ;
        const int64_t j0 = (int64_t)(pn.P0 + js - split * pn.nb) * BJ;
        float *seg = seg_min(a, (int)blockIdx.x, js);
        for (int o = 4 * ct; o < real; o += 4 * MAXCONS) {
            const float4 v = *reinterpret_cast<const float4 *>(sbest + o);
            const uint4 w = *reinterpret_cast<const uint4 *>(sruns + o);
            const float bb[4] = {v.x, v.y, v.z, v.w};
            const uint32_t r[4] = {w.x, w.y, w.z, w.w};
            float out[4];
#pragma unroll
            for (int x = 0; x < 4; x++) {
                out[x] = r[x] == kNoRuns ? CUDART_INF_F : bb[x];
                if (r[x] != kNoRuns) {
                    const int t = (o + x) / BJ, gl = t / L;
                    uint32_t w1 = (uint32_t)S.okey[r[x] & 0xFFu] << 16 | S.okey[(r[x] >> 8) & 0xFFu];
                    uint32_t w2 = r[x] >> 24 ? (uint32_t)S.okey[(r[x] >> 16) & 0xFFu] << 16 | S.okey[r[x] >> 24] : 0u;
                    if (next && __ldcg(seg + o + x) <= __fadd_rn(bb[x], __fmul_rn(bb[x], S.tau[3 + t - gl * L]))) {
                        const uint2 old = __ldcg(seg_runs(a, seg) + o + x);
                        uint32_t f1 = old.x, f2 = old.y;
                        bool any = true;
                        band_append(f1, f2, any, w1 >> 16, w1 & 0xFFFFu);
                        if (w2) band_append(f1, f2, any, w2 >> 16, w2 & 0xFFFFu);
                        w1 = f1;
                        w2 = f2;
                    }
                    __stcg(seg_runs(a, seg) + o + x, make_uint2(w1, w2));
                    atomicMin(reinterpret_cast<int *>(
                                  a.dp32 + d32(a, split * a.Gc + gl, 3 + t - gl * L, j0 + ((o + x) & (BJ - 1)))),
                              __float_as_int(bb[x]));
                }
            }
            if (next) {  // an output without tiles in this part keeps what it has
#pragma unroll
                for (int x = 0; x < 4; x++)
                    if (r[x] != kNoRuns) __stcg(seg + o + x, out[x]);
            } else __stcg(reinterpret_cast<float4 *>(seg + o), make_float4(out[0], out[1], out[2], out[3]));
        }
    };
    auto start = [&]() {
        const int split = js / pn.nb, Jl = js - split * pn.nb, real = min(a.Gc, a.G - split * a.Gc) * L * BJ;
        const int *u = ub_at(a, Jl, split * a.Gc);
        for (int o = 4 * ct; o < real; o += 4 * MAXCONS) {
            *reinterpret_cast<float4 *>(sbest + o) = far_start(a, u, pn.P0 + Jl, o);
            *reinterpret_cast<uint4 *>(sruns + o) = make_uint4(kNoRuns, kNoRuns, kNoRuns, kNoRuns);
        }
    };
    // the rows that hold the share's start and end may give it no task: their segments are empty
    auto empty = [&](int j) {
        float *seg = seg_min(a, (int)blockIdx.x, j);
        for (int o = ct; o < nt * BJ; o += MAXCONS) __stcg(seg + o, CUDART_INF_F);
    };
    const int js0 = S.first / pn.nB;
    if (ct == 0) { S.lnext = S.first; S.lpos = S.fpos; }
    uint32_t batch = 0;
    for (;;) {
        __syncthreads();  // the list before is done, its folds too
        far_list(a, S, pn);
        const int count = S.lcount;
        if (wid < 5 * min(count, kFarBufs)) {
            const int i = wid / 5;
            far_issue(a, S, big, pn, i, i, (int)((pp.n + (uint32_t)i) % kFarBufs), wid - 5 * i, policy);
        }
        for (int i = 0; i < count; i++) {
            const uint32_t key = S.lkey[i];
            const int jsn = (int)(key >> 14), K = (int)(key & 0x3FFFu), b = (int)(pp.n % kFarBufs), slot = i & 3;
            const uint4 bits = S.lbits[i];
            const int n = __popc(bits.x) + __popc(bits.y) + __popc(bits.z) + __popc(bits.w);
            if (jsn != js) {
                __syncthreads();  // the folds of the entry before are done
                if (js >= 0) flush();
                else if (jsn != js0) empty(js0);
                __syncthreads();
                js = jsn;
                ord = a.first_ord - 1;
                lastK = -2;
                next = false;
                start();
            }
            if (K != lastK) {
                cont = K == lastK + 1;
                if (++ord > kLastOrd) {
                    __syncthreads();  // the folds of the entry before are done
                    flush();
                    __syncthreads();
                    next = true;
                    ord = a.first_ord;
                    for (int o = ct; o < nt * BJ; o += MAXCONS) sruns[o] = kNoRuns;
                }
                if (ct == 0) S.okey[ord] = (uint16_t)K;
                lastK = K;
            }
            mbar_wait_bounded(&S.full[b], (pp.n / kFarBufs) & 1u, a.st, a.abort_flag);
            pp.n++;
            const float *buf = far_buf(a, big, b), *rows = buf + kCostTileFloats + 8 * slice;
            float4 C[2], F[2];
#pragma unroll
            for (int x = 0; x < 2; x++) {
                C[x] = *reinterpret_cast<const float4 *>(buf + col * PSTR + 8 * slice + 4 * x);
                F[x] = *reinterpret_cast<const float4 *>(buf + kCostHalfFloats + col * PSTR + 8 * slice + 4 * x);
            }
            for (int k0 = 0; k0 < n; k0 += kBatch, batch++) {
                int *pt = part + (int)(batch & 1u) * kBatch * 8 * BJ;
                // The tasks' multipliers come at once, and four tasks run as one block without a branch: the time of a tile
                // is the latency of such chains (a branch where the multiplier changes and the multiplier's loads in
                // every task's chain: 25.1 ms a pass at d = 2^17; the loads at once 23.5; now 22.5).  Tasks past
                // the entry's last leave slots that nothing reads.
#pragma unroll
                for (int h = 0; h < kBatch; h += 4) {
                    if (k0 + h >= n) break;
                    const float4 l4 = *reinterpret_cast<const float4 *>(&S.tlam[slot][k0 + h]);
                    const float lm[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                    for (int y = 0; y < 4; y++) {
                        const float4 p = *reinterpret_cast<const float4 *>(rows + (k0 + h + y) * BK);
                        const float4 q = *reinterpret_cast<const float4 *>(rows + (k0 + h + y) * BK + 4);
                        const float2 lam2 = make_float2(lm[y], lm[y]);
                        // candidates are >= +0, so their bits order like the values: integer mins
                        const float2 v0 = add2(make_float2(p.x, p.y), fma2(lam2, make_float2(F[0].x, F[0].y), make_float2(C[0].x, C[0].y)));
                        const float2 v1 = add2(make_float2(p.z, p.w), fma2(lam2, make_float2(F[0].z, F[0].w), make_float2(C[0].z, C[0].w)));
                        const float2 v2 = add2(make_float2(q.x, q.y), fma2(lam2, make_float2(F[1].x, F[1].y), make_float2(C[1].x, C[1].y)));
                        const float2 v3 = add2(make_float2(q.z, q.w), fma2(lam2, make_float2(F[1].z, F[1].w), make_float2(C[1].z, C[1].w)));
                        const int x0 = min(min(__float_as_int(v0.x), __float_as_int(v0.y)), __float_as_int(v1.x));
                        const int x1 = min(min(__float_as_int(v2.x), __float_as_int(v2.y)), __float_as_int(v3.x));
                        pt[((h + y) * 8 + slice) * BJ + col] = min(min(x0, x1), min(__float_as_int(v1.y), __float_as_int(v3.y)));
                    }
                }
                // (what the fold needs of its task, before the barrier)
                const int k = k0 + slice;
                const uint32_t f = k < n ? S.tinfo[slot][k] : 0u;
                const float tau = S.tau[3 + ((f >> 8) & 0xFFu)];
                __syncthreads();  // the batch's partial minima are complete
                // (the last batch: the tile's buffer is free, for the entry kFarBufs further on)
                if (k0 + kBatch >= n && i + kFarBufs < count && ((wid - 5 * i) & 15) < 5)
                    far_issue(a, S, big, pn, i + kFarBufs, (i + kFarBufs) & 3, b, (wid - 5 * i) & 15, policy);
                if (k < n) {
                    const int *pk = pt + slice * 8 * BJ + col;
                    int v = pk[0];
#pragma unroll
                    for (int x = 1; x < 8; x++) v = min(v, pk[x * BJ]);
                    const int o = (int)(f & 0xFFu) * BJ + col;
                    const float bb = sbest[o], T = __fmul_rn(bb, tau);
                    // a tile's minimum below bb - bb tau restarts the band, up to bb + bb tau joins it
                    // (band limits: the tests on the bits hold for bb = +inf too)
                    if ((uint32_t)v <= __float_as_uint(__fadd_rn(bb, T))) {
                        sruns[o] = runs_add(sruns[o], (uint32_t)v < __float_as_uint(__fsub_rn(bb, T)), (uint32_t)ord, cont);
                        sbest[o] = fminf(bb, __int_as_float(v));
                    }
                }
            }
            if (ct == 0) pp.run += (uint32_t)n;
            pp.fetched++;
        }
        if (!S.lmore) break;
    }
    __syncthreads();
    if (js >= 0) flush();
    else empty(js0);
    const int last = min(((int)blockIdx.x + 1) * S.share, S.total) - 1;
    int je = max(js, js0);
    while (je + 1 < pn.nb * a.nsplit && S.jstart[je + 1] <= last) je++;
    if (je > max(js, js0)) empty(je);
}

// ---------------------------------------------------------------- near phase
constexpr int kNearTiles = 4;   // tiles (K, J) of one J per CTA, consecutive K
constexpr int kNearMults = 2;   // multipliers per CTA
constexpr int kPanelMax = 16;   // column blocks per panel, at most (four groups of tiles per block)
// Groups of tiles of the blocks before Jl, and in a panel of nb blocks.
__host__ __device__ __forceinline__ int near_groups(int nb) {
    const int f = nb / kNearTiles, r = nb % kNearTiles;
    return kNearTiles * f * (f + 1) / 2 + r * (f + 1);
}
__device__ __forceinline__ int2 ld_relaxed2(const int *p) {
    int2 v;
    asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(int *p, int v) {
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Minima of tile group `grp` (near_groups(Jl) + group of Jl) and of single tiles, multiplier g: rows
// of 64 by layer index li = i - 3.
__device__ __forceinline__ int *near_group_min(const FastArgs &a, int grp, int g) {
    return a.tmin + ((size_t)grp * a.G + g) * (size_t)(a.s - 2) * BJ;
}
__device__ __forceinline__ int near_tile(int Kl, int Jl) { return Jl * (Jl + 1) / 2 + Kl; }
__device__ __forceinline__ float *near_tile_min(const FastArgs &a, int nt, int g) {
    return a.tmin1 + ((size_t)nt * a.G + g) * (size_t)(a.s - 2) * BJ;
}

// Row i >= 3 of block K = P0 + Kl at multiplier g, columns 2 lane and 2 lane + 1: the far
// minimum and the minima of the tile groups of block Kl, polled until each carries the panel's tag
// in its sign bit.  False when the wait gave up.
__device__ __forceinline__ bool near_gather(const FastArgs &a, int P0, int Kl, int g, int i, int tag, int lane, int &m0,
                                            int &m1) {
    const int2 far = ld_relaxed2(reinterpret_cast<const int *>(a.dp32 + d32(a, g, i, (int64_t)(P0 + Kl) * BJ + 2 * lane)));
    const int *src = near_group_min(a, near_groups(Kl), g) + (size_t)(i - 3) * BJ + 2 * lane;
    const size_t stride = (size_t)a.G * (size_t)(a.s - 2) * BJ;
    const int n = Kl / kNearTiles;  // groups 0..n
    uint32_t spins = 0;
    for (;;) {
        // every source at once: a poll is one round trip to L2, and the last writer ends it
        int bad = 0;
        m0 = far.x;
        m1 = far.y;
#pragma unroll
        for (int u = 0; u < kPanelMax / kNearTiles; u++)
            if (u <= n) {
                const int2 v = ld_relaxed2(src + u * stride);
                const int x = v.x ^ tag, y = v.y ^ tag;
                bad |= x | y;
                m0 = min(m0, x);
                m1 = min(m1, y);
            }
        if (!__any_sync(0xffffffffu, bad < 0)) return true;
        if ((++spins & 63u) == 0u) {
            int stop = 0;
            if (lane == 0) {
                stop = *(volatile int *)a.abort_flag;
                if (!stop && spins > a.spin_limit) {
                    a.st->timeout = 1;
                    atomicExch(a.abort_flag, 1);
                    stop = 1;
                }
            }
            if (__shfl_sync(0xffffffffu, stop, 0)) return false;
        }
    }
}

// A CTA's near item: tile group `grp` of block Jl (tiles 4 grp .. of it) and multipliers g0, g0 + 1.
struct NearItem { int Jl, grp, g0; };
__device__ __forceinline__ bool near_item(const FastArgs &a, int cta, int nb, NearItem &it) {
    const int pairs = (a.G + kNearMults - 1) / kNearMults;
    const int x = cta / pairs;
    if (x >= near_groups(nb)) return false;
    it.g0 = (cta - x * pairs) * kNearMults;
    int Jl = 0;
    while (near_groups(Jl + 1) <= x) Jl++;
    it.Jl = Jl;
    it.grp = x - near_groups(Jl);
    return true;
}

// The near phase of one panel; the item's cost tiles are in `tiles`, ex and rowbuf are scratch.  The
// diagonal tile's warp also writes the block's final dp32 rows, its block minima and last column
// (read by later panels' far phases).
static __device__ __noinline__ void near_phase(const FastArgs &a, Smem &S, const float *tiles, float *rowbuf, int P0,
                                               NearItem it, int tag) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, q = wid & 3, h = (wid >> 2) & 1, half = wid >> 3;
    const int g = it.g0 + h;
    if (g >= a.G) return;  // all eight warps of this multiplier
    const int Kl = it.grp * kNearTiles + q, K = P0 + Kl, J = P0 + it.Jl;
    const bool have = Kl <= it.Jl, diag = Kl == it.Jl;
    const float lam = S.lam32[g];
    const float2 lam2 = make_float2(lam, lam);
    const int col = lane + 32 * half;
    float2 W[BK / 2];  // costs of the lane's column
    const float *tile = tiles + (size_t)q * kCostTileFloats + col * PSTR;
#pragma unroll
    for (int kk = 0; kk < BK; kk += 4) {
        float4 c4 = make_float4(CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, CUDART_INF_F);
        float4 f4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (have) {
            c4 = *reinterpret_cast<const float4 *>(tile + kk);
            f4 = *reinterpret_cast<const float4 *>(tile + kCostHalfFloats + kk);
        }
        W[kk / 2] = fma2(lam2, make_float2(f4.x, f4.y), make_float2(c4.x, c4.y));
        W[kk / 2 + 1] = fma2(lam2, make_float2(f4.z, f4.w), make_float2(c4.z, c4.w));
    }
    float *row = rowbuf + wid * 2 * BK;
    int *ex = reinterpret_cast<int *>(rowbuf + (MAXCONS / 32) * 2 * BK) + h * 2 * kNearTiles * BJ;  // [parity][tile][64]
    const int oc = (q + 4 * half) * 8 + lane;  // lanes 0..7: the column whose group minimum this lane writes
    int *out = near_group_min(a, near_groups(it.Jl) + it.grp, g) + oc;
    float *out1 = near_tile_min(a, have ? near_tile(Kl, it.Jl) : 0, g) + col;
    const bool hold = a.hold0 && J == 0;  // test hook: block 0 is never published
    float *mdp = a.mdp + ((size_t)J * a.G + g) * a.mdp_stride, *dlast = a.dlast + ((size_t)J * a.G + g) * a.mdp_stride;
    bool dead = false;  // a wait gave up: only the barriers are kept
    for (int i = 3; i <= a.s; i++) {
        int m0 = 0x7f800000, m1 = 0x7f800000;  // row i - 1 of block K, columns 2 lane, 2 lane + 1
        if (have && !dead) {
            if (i == 3) {
                const int2 r = ld_relaxed2(reinterpret_cast<const int *>(a.dp32 + d32(a, g, 2, (int64_t)K * BK + 2 * lane)));
                m0 = r.x;
                m1 = r.y;
            } else if (!near_gather(a, P0, Kl, g, i - 1, tag, lane, m0, m1)) {
                dead = true;
            }
        }
        float *rw = row + (i & 1) * BK;
        *reinterpret_cast<float2 *>(rw + 2 * lane) = make_float2(__int_as_float(m0), __int_as_float(m1));
        __syncwarp();
        int a0 = 0x7f800000, a1 = 0x7f800000, b0 = 0x7f800000, b1 = 0x7f800000;
#pragma unroll
        for (int kk = 0; kk < BK; kk += 8) {
            const float4 d4 = *reinterpret_cast<const float4 *>(rw + kk), e4 = *reinterpret_cast<const float4 *>(rw + kk + 4);
            const float2 s0 = add2(make_float2(d4.x, d4.y), W[kk / 2]), s1 = add2(make_float2(d4.z, d4.w), W[kk / 2 + 1]);
            const float2 t0 = add2(make_float2(e4.x, e4.y), W[kk / 2 + 2]), t1 = add2(make_float2(e4.z, e4.w), W[kk / 2 + 3]);
            a0 = min(min(a0, __float_as_int(s0.x)), __float_as_int(s0.y));
            a1 = min(min(a1, __float_as_int(s1.x)), __float_as_int(s1.y));
            b0 = min(min(b0, __float_as_int(t0.x)), __float_as_int(t0.y));
            b1 = min(min(b1, __float_as_int(t1.x)), __float_as_int(t1.y));
        }
        a0 = min(min(a0, a1), min(b0, b1));
        int *x = ex + (i & 1) * kNearTiles * BJ;
        x[q * BJ + col] = a0;
        bar_sync(BAR_NEAR + h, 256);
        if (lane < 8 && !hold && !dead)
            st_relaxed(out + (size_t)(i - 3) * BJ,
                       min(min(x[oc], x[BJ + oc]), min(x[2 * BJ + oc], x[3 * BJ + oc])) ^ tag);
        if (have) out1[(size_t)(i - 3) * BJ] = __int_as_float(a0);
        if (diag && half == 0) {
            if (i > 3)
                *reinterpret_cast<float2 *>(a.dp32 + d32(a, g, i - 1, (int64_t)J * BJ + 2 * lane)) =
                    make_float2(__int_as_float(m0), __int_as_float(m1));
            const int mn = __reduce_min_sync(0xffffffffu, min(m0, m1));  // block minimum of row i - 1
            if (lane == 0) mdp[i - 3] = __int_as_float(mn);
            if (lane == 31) dlast[i - 3] = __int_as_float(m1);
        }
    }
    if (diag && half == 0 && !dead) {
        int m0, m1;
        if (near_gather(a, P0, Kl, g, a.s, tag, lane, m0, m1))
            *reinterpret_cast<float2 *>(a.dp32 + d32(a, g, a.s, (int64_t)J * BJ + 2 * lane)) =
                make_float2(__int_as_float(m0), __int_as_float(m1));
    }
}

// Band words of a panel's outputs from the far segments and the near tiles in increasing K: a
// segment (or tile) whose minimum lies above the output's band limit adds nothing; else its runs
// are appended as a walk appends tiles (runs_add).
static __device__ __noinline__ void fold_panel(const FastArgs &a, const Smem &S, const Panel &pn) {
    const int L = a.s - 2, per = a.G * L * BJ;
    for (int idx = (int)(blockIdx.x * MAXCONS + threadIdx.x); idx < pn.nb * per;
         idx += (int)(gridDim.x * MAXCONS)) {
        const int Jl = idx / per, o = idx - Jl * per;
        const int g = o / (L * BJ), li = (o / BJ) % L, jl = o & (BJ - 1);
        const int64_t j = (int64_t)(pn.P0 + Jl) * BJ + jl;
        if (j >= a.p) continue;
        const float m = __ldcg(a.dp32 + d32(a, g, 3 + li, j));
        const float lim = __fadd_rn(m, __fmul_rn(m, S.tau[3 + li]));
        uint32_t w1 = 0, w2 = 0;
        bool any = false;
        auto append = [&](uint32_t f, uint32_t l) { band_append(w1, w2, any, f, l); };
        if (pn.P0 > 0) {
            const int split = g / a.Gc, js = split * pn.nb + Jl;
            const int p0 = S.jstart[js], p1 = S.jstart[js + 1];
            if (p1 > p0) {
                const int c0 = p0 / S.share, c1 = (p1 - 1) / S.share;
                const size_t so = (size_t)(g - split * a.Gc) * L * BJ + (size_t)li * BJ + jl;
#pragma unroll 4
                for (int c = c0; c <= c1; c++) {
                    float *seg = seg_min(a, c, js);
                    if (__ldcg(seg + so) <= lim && m < CUDART_INF_F) {
                        const uint2 r = __ldcg(seg_runs(a, seg) + so);
                        append(r.x >> 16, r.x & 0xFFFFu);
                        if (r.y) append(r.y >> 16, r.y & 0xFFFFu);
                    }
                }
            }
        }
        const int *grp = near_group_min(a, near_groups(Jl), g) + (size_t)li * BJ + jl;
        const float *tm = near_tile_min(a, near_tile(0, Jl), g) + (size_t)li * BJ + jl;
        const size_t step = (size_t)per;
#pragma unroll
        for (int u = 0; u < kPanelMax / kNearTiles; u++) {
            if (u * kNearTiles > Jl) continue;
            if (!(__int_as_float(__ldcg(grp + u * step) & 0x7fffffff) <= lim)) continue;
            for (int Kl = u * kNearTiles; Kl <= min(Jl, u * kNearTiles + kNearTiles - 1); Kl++)
                if (__ldcg(tm + Kl * step) <= lim) append((uint32_t)(pn.P0 + Kl), (uint32_t)(pn.P0 + Kl));
        }
        a.band[oidx(a, g, 3 + li, j)] = band_pack(w1, w2);
    }
}

// The min-plus sweep over column blocks [J0, J1), panel by panel (see above).  build: the costs
// buffer holds one panel's tiles, computed here before the panel's far phase (no resident or
// streamed table).  Cooperative launch, one CTA of 512 threads per SM.
__global__ void __launch_bounds__(MAXCONS, 1) k_wavefront(const __grid_constant__ FastArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &S = *reinterpret_cast<Smem *>(smem_raw);
    float *big = reinterpret_cast<float *>(smem_raw + kSmemHead);
    const int ct = threadIdx.x;
    for (int q = ct; q <= kMaxS; q += MAXCONS) S.tau[q] = a.prm->tau[q];
    if (ct < kMaxG) S.lam32[ct] = a.prm->lam32[ct];
    if (ct < 32 * kTaskWords) S.tdiv[ct] = (uint16_t)(ct % (a.s - 2) | ct / (a.s - 2) << 8);
    if (ct == 0) {
        for (int b = 0; b < 2; b++) mbar_init(&S.smbar[b], 1);
        for (int b = 0; b < kFarBufs; b++) mbar_init(&S.full[b], 1 + kTaskWords);
        mbar_init(&S.nbar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    const uint64_t policy = policy_evict_first();
    Pipe pp{0u, 0u, 0u, 0u, 0u};
    int epoch = 0, panel = 0;
    bool ok = true;
    for (int P0 = a.J0; P0 < a.J1 && ok; P0 += a.T, panel++) {
        Panel pn;
        pn.P0 = P0;
        pn.nb = min(a.T, a.J1 - P0);
        pn.nB = (P0 + NT - 1) / NT;
        pn.tag = (panel & 1) ? (int)0x80000000 : 0;
        pn.tbase = a.build ? (size_t)P0 * (P0 + 1) / 2 : a.tile_base;
        if (a.build) {
            // (a tile is one long chain of 64 steps: 14 us, so six groups beside one another, the CTAs' first ones first)
            if (ct < kBuildGroups * NPROD)
                build_panel(a, reinterpret_cast<BuildSmem *>(big)[ct / NPROD], ct % NPROD, BAR_BUILD + ct / NPROD,
                            (int64_t)pn.tbase + ct / NPROD * gridDim.x + blockIdx.x, (int64_t)gridDim.x * kBuildGroups,
                            (int64_t)(P0 + pn.nb) * (P0 + pn.nb + 1) / 2, (int64_t)pn.tbase);
            ok = grid_sync(a, S, ++epoch);
            if (!ok) break;
        }
        if (P0 > 0) {
            if (a.bound) {
                bound_phase(a, S, big, pn, policy, pp.ns);
                ok = grid_sync(a, S, ++epoch);
                if (!ok) break;
            }
            mask_phase(a, S, big, pn, policy, pp.ns);
            ok = grid_sync(a, S, ++epoch);
            if (!ok) break;
            far_plan(a, S, pn);
            far_phase(a, S, big, pn, policy, pp);
            __syncthreads();  // the tile buffers are free
        }
        // this CTA's near tiles: their costs depend on nothing, so their copies overlap the barrier
        NearItem it{0, 0, 0};
        const bool near = near_item(a, (int)blockIdx.x, pn.nb, it);
        const int Kn0 = it.grp * kNearTiles, nk = near ? min(kNearTiles, it.Jl - Kn0 + 1) : 0;
        if (near && ct == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");
            mbar_expect_tx(&S.nbar, (uint32_t)nk * 2 * kCostHalfBytes);
            // consecutive K of one column block: one run of the table
            bulk_g2s(big, a.costs + (cost_tile_idx(P0 + Kn0, P0 + it.Jl) - pn.tbase) * kCostTileFloats,
                     (uint32_t)nk * 2 * kCostHalfBytes, &S.nbar, policy);
        }
        if (P0 > 0) ok = grid_sync(a, S, ++epoch);  // the panel's far minima are complete
        if (a.bound && ok) {  // the bounds were last read before this barrier: cleared for the next panel
            const int nn = a.T * a.G * (a.s - 2) * BJ;
            for (int q = (int)blockIdx.x * MAXCONS + ct; q < nn; q += (int)gridDim.x * MAXCONS) a.ub[q] = kNoBound;
        }
        if (near) {
            mbar_wait_bounded(&S.nbar, pp.nnear & 1u, a.st, a.abort_flag);
            pp.nnear++;
            pp.fetched += (uint32_t)nk;
            if (ct == 0)  // the tasks of the tiles below the diagonal
                pp.run += (uint32_t)(min(nk, it.Jl - Kn0) * min(kNearMults, a.G - it.g0) * (a.s - 2));
            if (ok) near_phase(a, S, big, big + kNearTiles * kCostTileFloats, P0, it, pn.tag);
        }
        if (!ok) break;
        ok = grid_sync(a, S, ++epoch, !(a.hold0 && blockIdx.x == 0));  // the panel's rows are final
        if (ok) fold_panel(a, S, pn);
    }
    if (ct == 0) atomicAdd(a.work, (unsigned long long)pp.run);
    if (ct == 0 && pp.fetched) atomicAdd((unsigned long long *)&a.st->tiles_fetched, (unsigned long long)pp.fetched);  // one cost tile per buffer fill
}

// ------------------------------------------------------------ base layer
// eq. apx_base for every multiplier: exact dp64, bp and the fp32 copy; all
// other rows cleared (dp64 = +inf, bp = -1, dp32 = +inf).
__global__ void k_fast_clear(double *dp64, int32_t *bp, float *dp32, size_t n) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) { dp64[i] = CUDART_INF; bp[i] = -1; dp32[i] = CUDART_INF_F; }
}

__global__ void k_fast_base(Prefix P, FastArgs a, double *dp64, int32_t *bp) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1;
    if (j >= P.p) return;
    double C, U, D;
    pair_exact(P, 0, j, C, U, D);
    double phi = phi_exact(P, U, D, true);
    for (int g = 0; g < a.G; g++) {
        double v = __dadd_rn(C, __dmul_rn(a.prm->lam64[g], phi));
        dp64[oidx(a, g, 2, j)] = v;
        bp[oidx(a, g, 2, j)] = 0;
        a.dp32[d32(a, g, 2, j)] = __fadd_rn(__double2float_rn(v * a.sc2), 0.0f);  // >= +0 (no -0)
    }
}

// ------------------------------------------------------------- extraction
// fp32 value of candidate k for output (g, i, j), bit-identical to the wavefront.
__device__ __forceinline__ float cand32(float dprev, float lam, float C, float Phi) {
    return __fadd_rn(dprev, __fmaf_rn(lam, Phi, C));
}

// Visit the candidates k of tile K for output (g, i, j) in the wavefront's fp32
// arithmetic (k descending) and call f(k, value) for every k with value <= thr.
template <typename F>
__device__ void visit_tile(const FastArgs &a, int g, int i, int64_t j, int64_t K, float thr, F &&f) {
    int64_t J = j / BJ, j0 = J * BJ, k0 = K * BK;
    float lam = a.prm->lam32[g];
    const float *prev = a.dp32 + d32(a, g, i - 1, k0) - k0;  // prev[k] for k in tile K
    if (a.costs) {
        // the wavefront's own interval costs, read back from the resident table
        const float *cr = a.costs + (cost_tile_idx(K, J) - a.tile_base) * kCostTileFloats + (size_t)(j - j0) * PSTR;
        const float *pr = cr + kCostHalfFloats;
        int64_t khi = (K == J) ? j - 1 : k0 + BK - 1;
        for (int64_t k = khi; k >= k0; k--) {
            const float v = cand32(prev[k], lam, cr[k - k0], pr[k - k0]);
            if (v <= thr) f(k, v);
        }
        return;
    }
    float vj = a.v[j];
    const float d_f = (float)a.d;
    Rec r;
    int64_t khi;
    float c, ph;
    if (K == J) {
        r = rec_empty();
        khi = j;  // state of the empty interval (j, j]
    } else {
        khi = k0 + BK - 1;
        rec_anchor(a, khi, j, r);  // any evaluation within the certified bound will do
        rec_emit(r, vj, a.v[khi], d_f, a.invd, c, ph);
        const float v = cand32(prev[khi], lam, c, ph);
        if (v <= thr) f(khi, v);
    }
    for (int64_t k = khi - 1; k >= k0; k--) {
        rec_step(r, vj, a.v[k + 1], a.wf[k + 1], __fsub_rn(a.v[k + 1], a.v[k]));
        rec_emit(r, vj, a.v[k], d_f, a.invd, c, ph);
        const float v = cand32(prev[k], lam, c, ph);
        if (v <= thr) f(k, v);
    }
}

// Tiles listed by a band word (band_pack), in increasing order.
template <typename F>
__device__ void visit_band(const FastArgs &a, int g, int i, int64_t j, uint64_t w, float thr, F &&f) {
    const uint32_t w1 = (uint32_t)w, w2 = (uint32_t)(w >> 32);
    for (uint32_t K = w1 >> 16; K <= (w1 & 0xFFFFu); K++) visit_tile(a, g, i, j, (int64_t)K, thr, f);
    if (w2)
        for (uint32_t K = w2 >> 16; K <= (w2 & 0xFFFFu); K++) visit_tile(a, g, i, j, (int64_t)K, thr, f);
}

// Tiles a band word spans (both runs).
__device__ __forceinline__ uint32_t band_tiles(uint64_t w) {
    const uint32_t w1 = (uint32_t)w, w2 = (uint32_t)(w >> 32);
    return (w1 & 0xFFFFu) - (w1 >> 16) + 1u + (w2 ? (w2 & 0xFFFFu) - (w2 >> 16) + 1u : 0u);
}

__device__ __forceinline__ float band_threshold(const FastArgs &a, int i, float m32) {
    return __fadd_rn(m32, __fmul_rn(m32, a.prm->tau[i]));
}

// The candidates of output (g, i, j)'s band, by the 32 lanes of a warp together, with
// visit_tile's decisions (fp32 value <= thr): f(in, k, v) is called by every lane at once
// (a warp-uniform call; `in` is false for a lane without a candidate in that step;
// `v` is the candidate's fp32 value, +inf for a lane without one).
// With resident costs the lanes split every tile's k (the table gives any pair
// directly); otherwise they take whole tiles and walk them in step along visit_tile's
// recurrence (k descending from the anchor at the tile's top pair, or from the empty
// interval (j, j] on the diagonal tile), so the values, and the decisions, are visit_tile's.
template <typename F>
__device__ __forceinline__ void warp_visit_band(const FastArgs &a, int g, int i, int64_t j, uint64_t w, float thr,
                                                F &&f) {
    const int lane = threadIdx.x & 31;
    const uint32_t w1 = (uint32_t)w, w2 = (uint32_t)(w >> 32);
    const uint32_t n1 = (w1 & 0xFFFFu) - (w1 >> 16) + 1u;
    const uint32_t ntile = n1 + (w2 ? (w2 & 0xFFFFu) - (w2 >> 16) + 1u : 0u);
    const float lam32 = a.prm->lam32[g];
    const int64_t J = j / BJ, j0 = J * BJ;
    if (a.costs) {
        for (uint32_t t = 0; t < ntile; t++) {
            const int64_t K = t < n1 ? (w1 >> 16) + t : (w2 >> 16) + (t - n1);
            const int64_t k0 = K * BK;
            const float *cr = a.costs + (cost_tile_idx(K, J) - a.tile_base) * kCostTileFloats + (size_t)(j - j0) * PSTR;
            const float *pr = cr + kCostHalfFloats;
            const float *prev32 = a.dp32 + d32(a, g, i - 1, k0) - k0;
            const int64_t khi = (K == J) ? j - 1 : k0 + BK - 1;
            for (int64_t kb = k0; kb <= khi; kb += 32) {  // warp-uniform
                const int64_t k = kb + lane;
                const float v = k <= khi ? cand32(prev32[k], lam32, cr[k - k0], pr[k - k0]) : CUDART_INF_F;
                f(v <= thr, k, v);
            }
        }
        return;
    }
    const float vj = a.v[j], d_f = (float)a.d;
    for (uint32_t tb = 0; tb < ntile; tb += 32) {  // warp-uniform
        const uint32_t t = tb + lane;
        // tile K of the band (lanes past the band's end take tile 0 and no candidate)
        const int64_t K = t >= ntile ? 0 : (int64_t)(t < n1 ? (w1 >> 16) + t : (w2 >> 16) + (t - n1));
        const int64_t k0 = K * BK;
        const float *prev32 = a.dp32 + d32(a, g, i - 1, k0) - k0;
        Rec r = rec_empty();
        int64_t kfirst = k0 + BK - 1;
        int nk = 0;  // candidates of the lane's tile: k = kfirst, kfirst - 1, ..., kfirst - nk + 1
        if (t < ntile) {
            if (K == J) {
                kfirst = j - 1;
                nk = (int)(j - k0);
            } else {
                nk = BK;
                rec_anchor(a, kfirst, j, r);
            }
        }
        for (int it = 0; it < BK; it++) {  // warp-uniform
            const int64_t k = kfirst - it;
            float v = CUDART_INF_F;
            if (it < nk) {
                if (it > 0 || K == J) rec_step(r, vj, a.v[k + 1], a.wf[k + 1], __fsub_rn(a.v[k + 1], a.v[k]));
                float c, ph;
                rec_emit(r, vj, a.v[k], d_f, a.invd, c, ph);
                v = cand32(prev32[k], lam32, c, ph);
            }
            f(it < nk && v <= thr, k, v);
        }
    }
}

// Outputs eq. apx_final reads: dp(i, p-1) for i in [ilo, s] (mode kNeedFinal), or every output (kNeedAll).  A pass of
// the multiplier search, whose tables nobody reads, needs only the layers whose fp32 value is within the
// band of the least one (kNeedLeast): another layer's exact value is above the least exact one, and so is the fp32
// value that its table entry keeps.  Usually that is one layer, and its closure a chain instead of s - 2 of them:
// the need and exact stages of a pass take 2.1 instead of 4.8 ms at d = 50001, s = 32.
// The first thread also turns the pass's task count into (multiplier, tile) units of s - 2 tasks.
enum NeedMode { kNeedFinal, kNeedAll, kNeedLeast };
__global__ void k_need_init(FastArgs a, int ilo, NeedMode mode) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t units = (int64_t)a.G * a.nJ * (a.nJ - 1) / 2, run = (int64_t)*a.work / (a.s - 2);
        a.st->tiles_run += run;
        a.st->tiles_skipped += max((int64_t)0, units - run);
    }
    int64_t tot = (int64_t)a.G * (a.s + 1) * a.ps;
    int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; id < tot; id += stride) {
        int64_t j = id % a.ps;
        int i = (int)((id / a.ps) % (a.s + 1));
        uint8_t v = 0;
        if (i >= 3 && j < a.p && j >= i - 1) v = mode == kNeedAll ? 1 : (j == a.p - 1 && i >= ilo);
        if (v && mode == kNeedLeast) {
            const int g = (int)(id / a.ps / (a.s + 1));
            float m = CUDART_INF_F;
            for (int l = ilo; l <= a.s; l++) m = fminf(m, a.dp32[d32(a, g, l, j)]);
            v = !(a.dp32[d32(a, g, i, j)] > __fadd_rn(m, __fmul_rn(m, a.prm->tau[a.s])));
        }
        a.need[id] = v;
    }
}

// Warp-aggregated append of `v` to list[*cnt] by the lanes of `mask` that want it.
__device__ __forceinline__ void warp_append(unsigned mask, bool want, int32_t v, int32_t *list, int *cnt) {
    const unsigned m = __ballot_sync(mask, want);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(mask, base, leader);
    if (want) list[base + __popc(m & ((1u << lane) - 1u))] = v;
}

__device__ __forceinline__ int32_t *layer_list(const FastArgs &a, int i, int kind) {
    return a.lists + ((size_t)i * 2 + kind) * (size_t)a.G * (size_t)a.ps;
}

// Backward closure, layer i: members of every needed output; mark (i-1, k) needed;
// list the needed outputs for the exact stage (inline members / big bands).  A thread
// walks an output's band when it spans at most kThreadTiles tiles; wider bands go to
// k_need_wide, a warp each (threads of one warp walking bands of very different widths
// would wait on the widest).  (Not in a pass that needs few outputs: k_need_wide<true>.)
constexpr uint32_t kThreadTiles = 4;
__global__ void k_need_layer(FastArgs a, int i) {
    if (*(volatile const int *)a.abort_flag) return;  // a wait gave up: the tables are not valid
    const int64_t tot = (int64_t)a.G * a.p;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long nmem = 0, nbig = 0;
    int32_t *lsmall = layer_list(a, i, 0), *lbig = layer_list(a, i, 1);
    int *csmall = a.list_cnt + 2 * i, *cbig = csmall + 1;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < tot; base += stride) {  // warp-uniform trip count
        const int64_t id = base + threadIdx.x;
        bool listed = false, wide = false;
        int cnt = 0;
        int32_t packed = 0;
        if (id < tot) {
            const int64_t j = id % a.p;
            const int g = (int)(id / a.p);
            const size_t o = oidx(a, g, i, j);
            if (j >= i - 1 && a.need[o]) {
                const float m32 = a.dp32[d32(a, g, i, j)];
                if (!(m32 < CUDART_INF_F)) {
                    a.mcnt[o] = 0;
                } else {
                    const uint64_t w = a.band[o];
                    packed = (int32_t)((g << 24) | (int32_t)j);
                    if (band_tiles(w) > kThreadTiles) {
                        wide = true;  // a warp walks it (k_need_wide): lanes' walks would diverge
                    } else {
                        int32_t *mem = a.members + o * NMEM;
                        uint8_t *below = a.need + oidx(a, g, i - 1, 0);
                        const bool mark = i - 1 >= 3;
                        float vmin = CUDART_INF_F;
                        int32_t kmin = -1;
                        visit_band(a, g, i, j, w, band_threshold(a, i, m32), [&](int64_t k, float v) {
                            if (cnt < NMEM) mem[cnt] = (int32_t)k;
                            cnt++;
                            if (mark) below[k] = 1;
                            if (v < vmin || (v == vmin && (int32_t)k < kmin)) { vmin = v; kmin = (int32_t)k; }
                        });
                        if (cnt > NMEM) mem[0] = kmin;  // a big output keeps its fp32 argmin (exact_big)
                        a.mcnt[o] = cnt;
                        nmem += cnt;
                        nbig += cnt > NMEM;
                        listed = true;
                    }
                }
            }
        }
        warp_append(0xffffffffu, listed && cnt <= NMEM, packed, lsmall, csmall);
        warp_append(0xffffffffu, listed && cnt > NMEM, packed, lbig, cbig);
        warp_append(0xffffffffu, wide, packed, a.wide, a.wide_cnt + i);
    }
    if (nmem) atomicAdd((unsigned long long *)&a.st->members, nmem);
    if (nbig) atomicAdd((unsigned long long *)&a.st->big_bands, nbig);
}

// The closure of layer i for the outputs k_need_layer deferred: a warp per output walks
// its band (warp_visit_band), marks (i-1, k) needed for every member, keeps the first
// NMEM members it meets (the exact stage's rule is order-free) and lists the output.
// CHAIN: for all outputs of the layer, those k_need_init marked and those on the chain's list, to which the layer above
// appended each output that it marked first; so a layer takes one launch and no pass over the marks (with
// k_need_layer 11 us a layer at d = 50001, s = 32, and 20 where its threads walked the bands; now 6).
__device__ __forceinline__ int32_t *chain_list(const FastArgs &a, int i) { return layer_list(a, i & 1, 0); }  // (layers 0, 1: free)
template <bool CHAIN>
__global__ void __launch_bounds__(128) k_need_wide(FastArgs a, int i) {
    if (*(volatile const int *)a.abort_flag) return;  // a wait gave up: the tables are not valid
    const int n = a.wide_cnt[i];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int warps = gridDim.x * (blockDim.x >> 5);
    const bool mark = i - 1 >= 3;
    int32_t *lsmall = layer_list(a, i, 0), *lbig = layer_list(a, i, 1);
    int *csmall = a.list_cnt + 2 * i, *cbig = csmall + 1;
    unsigned long long nmem = 0, nbig = 0, nover = 0;  // lane 0
    for (int e = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; e < n + (CHAIN ? a.G : 0); e += warps) {
        const int32_t v = !CHAIN ? a.wide[e] : e < n ? chain_list(a, i)[e] : (int32_t)((e - n) << 24 | (int)(a.p - 1));
        const int g = v >> 24;
        const int64_t j = v & 0xFFFFFF;
        const size_t o = oidx(a, g, i, j);
        if (CHAIN && e >= n && !a.need[o]) continue;  // no member is ever p - 1: not on the list too
        const float m32 = a.dp32[d32(a, g, i, j)];
        if (CHAIN && !(m32 < CUDART_INF_F)) {
            if (lane == 0) a.mcnt[o] = 0;
            continue;
        }
        const uint64_t w = a.band[o];
        int32_t *mem = a.members + o * NMEM;
        uint8_t *below = a.need + oidx(a, g, i - 1, 0);
        int cnt = 0;  // warp-uniform
        float vmin = CUDART_INF_F;  // per lane: its least member value, lowest k on ties
        int32_t kmin = INT32_MAX;
        warp_visit_band(a, g, i, j, w, band_threshold(a, i, m32), [&](bool in, int64_t k, float v) {
            const unsigned mask = __ballot_sync(0xffffffffu, in);
            bool fresh = false;
            if (in) {
                const int pos = cnt + __popc(mask & lt);
                if (pos < NMEM) mem[pos] = (int32_t)k;
                if (mark && CHAIN) {
                    const size_t at = oidx(a, g, i - 1, k);
                    const uint32_t bit = 1u << (8 * (at & 3));
                    fresh = !(atomicOr(reinterpret_cast<uint32_t *>(a.need + (at & ~(size_t)3)), bit) & bit);
                } else if (mark) below[k] = 1;
                if (v < vmin || (v == vmin && (int32_t)k < kmin)) { vmin = v; kmin = (int32_t)k; }
            }
            if (CHAIN && mark)
                warp_append(0xffffffffu, fresh, (int32_t)((g << 24) | (int32_t)k), chain_list(a, i - 1), a.wide_cnt + i - 1);
            cnt += __popc(mask);
        });
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float v2 = __shfl_xor_sync(0xffffffffu, vmin, off);
            const int32_t k2 = __shfl_xor_sync(0xffffffffu, kmin, off);
            if (v2 < vmin || (v2 == vmin && k2 < kmin)) { vmin = v2; kmin = k2; }
        }
        __syncwarp();  // every lane's member stores are done before lane 0 overwrites slot 0
        if (lane == 0) {
            if (cnt > NMEM) mem[0] = kmin;  // a big output keeps its fp32 argmin (exact_big)
            a.mcnt[o] = cnt;
            nmem += cnt;
            nbig += cnt > NMEM;
            nover += band_tiles(w) > 32u ? 1 : 0;  // wide bands (diagnostic)
            if (cnt <= NMEM) lsmall[atomicAdd(csmall, 1)] = v;
            else lbig[atomicAdd(cbig, 1)] = v;
        }
        __syncwarp();
    }
    if (lane == 0) {
        if (nmem) atomicAdd((unsigned long long *)&a.st->members, nmem);
        if (nbig) atomicAdd((unsigned long long *)&a.st->big_bands, nbig);
        if (nover) atomicAdd((unsigned long long *)&a.st->overflow, nover);
    }
}

// Outputs the answer does not read keep their fp32 minimum: dp64 = m32, bp = -2.
__global__ void k_fill_unneeded(FastArgs a, double *dp64, int32_t *bp) {
    if (*(volatile const int *)a.abort_flag) return;  // a wait gave up: the tables are not valid
    const int64_t tot = (int64_t)a.G * (a.s + 1) * a.ps;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < tot; o += stride) {
        const int64_t j = o % a.ps;
        const int i = (int)((o / a.ps) % (a.s + 1));
        const int g = (int)(o / (a.ps * (a.s + 1)));
        if (i < 3 || j >= a.p || j < i - 1 || a.need[o]) continue;
        const float m32 = a.dp32[d32(a, g, i, j)];
        if (m32 < CUDART_INF_F) { dp64[o] = (double)m32 * a.isc2; bp[o] = -2; }
    }
}

// ----------------------------------------------------------- exact layer
__device__ __forceinline__ double exact_value(const Prefix &P, const double *prev, int64_t k, int64_t j, double lam) {
    double C, U, D;
    pair_exact(P, k, j, C, U, D);
    return __dadd_rn(prev[k], __dadd_rn(C, __dmul_rn(lam, phi_exact(P, U, D, false))));
}
__device__ __forceinline__ void exact_candidate(const Prefix &P, const double *prev, int64_t k, int64_t j,
                                                double lam, double &best, int32_t &arg) {
    const double c = exact_value(P, prev, k, j, lam);
    if (c < best || (c == best && k < arg)) { best = c; arg = (int32_t)k; }
}

// Result of a resolved output and its certificate check: the fp32 minimum must lie
// within eps_i of the exact one.
__device__ __forceinline__ bool exact_store(const FastArgs &a, int g, int i, int64_t j, double best, int32_t arg,
                                            double *dp64, int32_t *bp) {
    const size_t o = oidx(a, g, i, j);
    dp64[o] = best;
    bp[o] = arg == INT32_MAX ? -1 : arg;
    const float m32 = a.dp32[d32(a, g, i, j)];
    const double e = (double)a.prm->eps[i], x = best * a.sc2;
    return fabs((double)m32 - x) <= e * x * 1.0001;
}

__device__ __forceinline__ void count_exact(const FastArgs &a, unsigned long long nres, int nviol) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nres += __shfl_xor_sync(0xffffffffu, nres, o);
        nviol += __shfl_xor_sync(0xffffffffu, nviol, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (nres) atomicAdd((unsigned long long *)&a.st->rescored, nres);
        if (nviol) atomicAdd(&a.st->bound_viol, nviol);
    }
}

// Layer i, outputs with at most NMEM members: one thread each, binary64 re-scoring
// with double-double interval costs; the lowest k among exact minima wins.
constexpr int kExactBlocks = 8, kExactBigBlocks = 16;  // blocks per SM
static __device__ __forceinline__ void exact_small(const Prefix &P, const FastArgs &a, int i, double *dp64, int32_t *bp, int block) {
    const int blocks = gridDim.x / (kExactBlocks + kExactBigBlocks) * kExactBlocks;
    // A warp takes up to 32 listed outputs at a time and evaluates their members flattened
    // (member r of the outputs' lists goes to lane r mod 32), so every lane of a
    // binary64 sequence does useful work; then each output's lane takes the least value,
    // lowest k on ties, over its own members (the per-output rule, which is order-free).
    // A short list is dealt to one warp on every SM (a sequence is 3 us of an SM's binary64 pipe, and 32
    // outputs a warp, four warps a block, put a few hundred outputs' on three SMs: 33 us a layer at
    // d = 50001, s = 32, now 13).
    __shared__ double sval[4][32 * NMEM];
    __shared__ int32_t sk[4][32 * NMEM];
    const int n = a.list_cnt[2 * i];
    const int32_t *list = layer_list(a, i, 0);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long nres = 0;
    int nviol = 0;
    const int nsm = blocks / kExactBlocks, per = min(32, (n + nsm - 1) / nsm);
    const int wstride = blocks * (blockDim.x >> 5) * per;
    for (int base = (wid * blocks + block) * per; base < n; base += wstride) {  // warp-uniform
        const int e = lane < per ? base + lane : n;
        int g = 0, cnt = 0;
        int64_t j = 0;
        long long o = 0;
        if (e < n) {
            const int32_t v = list[e];
            g = v >> 24;
            j = v & 0xFFFFFF;
            o = (long long)oidx(a, g, i, j);
            cnt = a.mcnt[o];
        }
        int off = cnt;  // inclusive, then exclusive prefix of the member counts
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, off, d);
            if (lane >= d) off += t;
        }
        const int total = __shfl_sync(0xffffffffu, off, 31);
        off -= cnt;
        for (int rb = 0; rb < total; rb += 32) {  // warp-uniform
            const int r = rb + lane;
            int ow = 0;  // the last lane whose offset is <= r: the owner of member r
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const int oc = __shfl_sync(0xffffffffu, off, ow + st);
                if (oc <= r) ow += st;
            }
            const int og = __shfl_sync(0xffffffffu, g, ow);
            const int64_t oj = __shfl_sync(0xffffffffu, j, ow);
            const long long oo = __shfl_sync(0xffffffffu, o, ow);
            const int q = r - __shfl_sync(0xffffffffu, off, ow);
            if (r < total) {
                const int32_t k = a.members[(size_t)oo * NMEM + q];
                sk[wid][r] = k;
                sval[wid][r] = exact_value(P, dp64 + oidx(a, og, i - 1, 0), k, oj, a.prm->lam64[og]);
            }
        }
        __syncwarp();
        if (cnt > 0) {
            double best = CUDART_INF;
            int32_t arg = INT32_MAX;
            for (int q = 0; q < cnt; q++) {
                const double c = sval[wid][off + q];
                const int32_t k = sk[wid][off + q];
                if (c < best || (c == best && k < arg)) { best = c; arg = k; }
            }
            nres += cnt;
            nviol += exact_store(a, g, i, j, best, arg, dp64, bp) ? 0 : 1;
        } else if (e < n) {
            nviol += exact_store(a, g, i, j, CUDART_INF, INT32_MAX, dp64, bp) ? 0 : 1;
        }
        __syncwarp();  // the staging slots are free for the next 32 outputs
    }
    count_exact(a, nres, nviol);
}

// Layer i, outputs with more members: one warp each (fp32 re-evaluation within the
// band by warp_visit_band, whose decisions are the closure stage's; exact re-scoring of
// the members met), then the lanes' results meet (value, then lowest k).  The members
// met wait in the warp's queue, and each time it holds 32 every lane re-scores one of
// them in binary64, so the binary64 sequence runs with all lanes busy (the result,
// least value then lowest k, does not depend on the order).
static __device__ __forceinline__ void exact_big(const Prefix &P, const FastArgs &a, int i, double *dp64, int32_t *bp, int block) {
    const int blocks = gridDim.x / (kExactBlocks + kExactBigBlocks) * kExactBigBlocks;
    __shared__ int32_t queue[4][32];  // per warp: band members waiting for binary64 re-scoring
    const int n = a.list_cnt[2 * i + 1];
    const int32_t *list = layer_list(a, i, 1);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int32_t *qw = queue[threadIdx.x >> 5];
    const int warps = blocks * (blockDim.x >> 5);
    unsigned long long nres = 0;
    int nviol = 0;
    for (int e = (threadIdx.x >> 5) * blocks + block; e < n; e += warps) {
        const int32_t v = list[e];
        const int g = v >> 24;
        const int64_t j = v & 0xFFFFFF;
        const size_t o = oidx(a, g, i, j);
        const float m32 = a.dp32[d32(a, g, i, j)];
        const float thr = band_threshold(a, i, m32);
        const uint64_t w = a.band[o];
        const double lam = a.prm->lam64[g];
        const double *prev = dp64 + oidx(a, g, i - 1, 0);
        double best = CUDART_INF;
        int32_t arg = INT32_MAX;
        int qn = 0;  // warp-uniform queue length
        // The closure stage kept the band's fp32 argmin kb in the member slot 0; its binary64
        // value b0 bounds the binary64 minimum from above.  Every fp32 candidate value is within
        // eps_i (relative) of the candidate's exact (real) value V, so V >= val32 / (1 + eps_i);
        // a binary64 candidate is within far less than 2^-40 of V (a few correctly rounded
        // operations per layer on non-negative terms, s <= 256 layers).  So a member with
        // val32 > b0 (1 + eps_i + 2^-30) has V > b0 (1 + 2^-31) and a binary64 value above b0:
        // it can neither be the minimum nor tie it, and is not re-scored.
        const int32_t kb = a.members[o * NMEM];
        double b0 = CUDART_INF;
        if (lane == 0 && kb >= 0) b0 = exact_value(P, prev, kb, j, lam);
        b0 = __shfl_sync(0xffffffffu, b0, 0);
        if (lane == 0 && kb >= 0) { best = b0; arg = kb; nres++; }
        const float thr2 = b0 < CUDART_INF
                               ? __double2float_ru(__dmul_ru(b0 * a.sc2, __dadd_ru(1.0 + 0x1p-30, (double)a.prm->eps[i])))
                               : CUDART_INF_F;
        warp_visit_band(a, g, i, j, w, thr, [&](bool in0, int64_t k, float v) {
            const bool in = in0 && v <= thr2 && (int32_t)k != kb;
            const unsigned mask = __ballot_sync(0xffffffffu, in);
            if (!mask) return;
            const int cnt = __popc(mask), pos = qn + __popc(mask & lt);
            if (in && pos < 32) qw[pos] = (int32_t)k;
            __syncwarp();
            if (qn + cnt >= 32) {
                exact_candidate(P, prev, qw[lane], j, lam, best, arg);
                nres++;
                __syncwarp();
                if (in && pos >= 32) qw[pos - 32] = (int32_t)k;
                __syncwarp();
                qn += cnt - 32;
            } else {
                qn += cnt;
            }
        });
        if (lane < qn) {
            exact_candidate(P, prev, qw[lane], j, lam, best, arg);
            nres++;
        }
        __syncwarp();  // the queue is free for the warp's next output
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double b2 = __shfl_xor_sync(0xffffffffu, best, off);
            const int32_t a2 = __shfl_xor_sync(0xffffffffu, arg, off);
            if (b2 < best || (b2 == best && a2 < arg)) { best = b2; arg = a2; }
        }
        if (lane == 0) nviol += exact_store(a, g, i, j, best, arg, dp64, bp) ? 0 : 1;
    }
    count_exact(a, nres, nviol);
}

// Layer i: the first blocks take the outputs with more members, the others the rest (one launch a layer).
__global__ void __launch_bounds__(128) k_exact_layer(Prefix P, FastArgs a, int i, double *dp64, int32_t *bp) {
    if (*(volatile const int *)a.abort_flag) return;  // a wait gave up: the tables are not valid
    const int big = gridDim.x / (kExactBlocks + kExactBigBlocks) * kExactBigBlocks;
    if ((int)blockIdx.x < big) exact_big(P, a, i, dp64, bp, (int)blockIdx.x);
    else exact_small(P, a, i, dp64, bp, (int)blockIdx.x - big);
}

// ------------------------------------------------------------------ host
// The values times sc (exact but below 2^-126); narrow: two of them end up too close for fp32 intervals.
__global__ void k_scale_values(const float *v, float *out, int64_t p, double sc, int *narrow) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p) return;
    const float x = (float)((double)v[i] * sc);
    out[i] = x;
    if (i > 0 && !(__fsub_rn(x, (float)((double)v[i - 1] * sc)) >= 0x1p-100f)) *narrow = 1;
}

__global__ void k_weights_f32(const int64_t *w, float *wf, int64_t p) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < p) wf[i] = (float)w[i];
}

// One word a thread (a single thread's copy took 9.7 us).
__global__ void k_store_params(FastParams prm, FastParams *dst) {
    static_assert(sizeof(FastParams) % 4 == 0, "copied by words");
    for (int i = threadIdx.x; i < (int)(sizeof(FastParams) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(dst)[i] = reinterpret_cast<const uint32_t *>(&prm)[i];
}

static int mdp_stride(int s) { return (s + 1 + 3) & ~3; }

// The band region: band words, need marks, flags (barrier, abort), constants, corner
// states, block minima, list counts; member counts and lists (scratch of the wavefront before the
// need stage writes them: scratch_bytes); then the seed rows (far_start).
static size_t flags_bytes(int64_t d) { return align256(8 * (size_t)kMaxG * (size_t)cdiv(d, BJ) + 64); }
// For 3 <= s < 6 as much as for s = 6: without a cost table a panel's tiles go there, 552 d bytes a column block, and the lists of
// three to five layers left room for two or three blocks a panel; the panels' barriers and tile chains then made a
// budgeted search slower than whole column blocks had (d = 12000, s = 3: 36 ms against 26; with four blocks 18).
constexpr int kScratchS = 6;
static size_t scratch_bytes(int64_t d, int32_t s) {
    const size_t rows = (size_t)kMaxG * (size_t)((s < 3 ? s : std::max(s, kScratchS)) + 1) * (size_t)table_stride(d);
    return align256(4 * rows) + align256(4 * NMEM * rows) + align256(2 * 4 * rows) +
           align256(4 * (size_t)kMaxG * (size_t)table_stride(d));
}
static size_t band_core_bytes(int64_t d, int32_t s) {
    size_t rows = (size_t)kMaxG * (size_t)(s + 1) * (size_t)table_stride(d);
    size_t nJ = (size_t)cdiv(d, BJ);
    return align256(8 * rows) + align256(rows) + flags_bytes(d) + align256(sizeof(FastParams)) +
           align256(32 * nJ * (nJ + 1) / 2) + align256(4 * (size_t)kMaxG * (size_t)mdp_stride(s) * nJ) +
           align256(4 * 2 * (size_t)(s + 1)) + align256(4 * (size_t)(s + 1)) + scratch_bytes(d, s);
}
static size_t seed_rows_bytes(int64_t d, int32_t s) { return align256(4 * (size_t)cdiv(d, BJ) * BJ * (size_t)(s + 1)); }
size_t fast_dp_band_bytes(int64_t d, int32_t s) { return band_core_bytes(d, s) + seed_rows_bytes(d, s); }
static float *seed_rows(void *ws, const Layout &Lw) {
    return reinterpret_cast<float *>(wsp<char>(ws, Lw.band) + band_core_bytes(Lw.d, Lw.s));
}

// Keep the fp32 dp rows of multiplier g of the last pass (G multipliers over p values) as
// the seed rows of a later pass at multipliers <= this one's (far_start).
int save_dp_seed(void *ws, const Layout &Lw, int64_t p, int G, int s, int g, cudaStream_t st) {
    if (g < 0 || g >= G || s != Lw.s) return ECASQ_EINVAL;
    const size_t row = (size_t)(s + 1) * BJ * sizeof(float);
    const float *src = wsp<float>(ws, Lw.dp32) + (size_t)g * (s + 1) * BJ;
    ECASQ_CUDA_TRY(cudaMemcpy2DAsync(seed_rows(ws, Lw), row, src, row * (size_t)G, row, (size_t)cdiv(p, BJ),
                                     cudaMemcpyDeviceToDevice, st));
    return ECASQ_OK;
}

static void band_factors(int s, FastParams &fp) { band_factors(s, fp.tau, fp.eps); }

// The resident table: every tile's C and Phi rows, then every tile's column summary
// (BJ float2), both indexed by J(J+1)/2 + K with J < ceil(d / 64).
size_t resident_costs_bytes(int64_t d) {
    if (d < 1) return 0;
    double nJ = (double)cdiv(d, BJ);
    double bytes = nJ * (nJ + 1.0) * 0.5 * ((double)kCostTileFloats * sizeof(float) + BJ * sizeof(float2));
    if (!(bytes < 9.0e18)) return 0;
    size_t n = (size_t)cdiv(d, BJ);
    return n * (n + 1) / 2 * (kCostTileFloats * sizeof(float) + BJ * sizeof(float2));
}

// Streamed interval costs: the cost tiles of a band of column blocks at a time, in a
// buffer of streamed_costs_bytes(d) (tiles, then their column summaries).  The band
// holds up to 64 full columns of tiles, so a band near the end of the triangle still
// has 64 blocks (times the multiplier splits) to spread over the SMs.
static size_t tile_bytes_with_summary() { return kCostTileFloats * sizeof(float) + BJ * sizeof(float2); }
size_t streamed_costs_bytes(int64_t d) {
    if (d < 1) return 0;
    const size_t nJ = (size_t)cdiv(d, BJ);
    const size_t full = nJ * (nJ + 1) / 2, band = std::min(full, (size_t)64 * nJ);
    return band * tile_bytes_with_summary();
}

// Scratch of the wavefront (member counts and lists, unused until the need stage): the blocks'
// last columns, the near minima, the bounds, the far lists, the far segments and, without a cost
// table, one panel's cost tiles.  Panels of T column blocks, as many as the GPU's SMs take near items
// of and as leave the scratch enough segments to spread a panel's far tiles over the SMs.
// Tiles of T column blocks, at most: those of the last ones.
static size_t panel_tiles(int T, int nJ) { return (size_t)T * nJ - (size_t)T * (T - 1) / 2; }
struct PanelPlan { int T, workers; size_t dlast, tmin, tmin1, ub, lists, part, costs; };
static bool plan_panels(size_t scratch, int nsm, int nJ, int G, int Gc, int nsplit, int s, bool build, PanelPlan *pl) {
    const size_t out = (size_t)G * (s - 2) * BJ;  // outputs of a column block
    const size_t seg = (size_t)Gc * (s - 2) * BJ * 12;
    const int pairs = (int)cdiv(G, kNearMults);
    int T = 1;
    while (T < kPanelMax && near_groups(T + 1) * pairs <= nsm) T++;
    if (near_groups(T) * pairs > nsm) return false;
    for (T = std::min(T, nJ); T >= 1; T--) {
        size_t off = 0;
        auto take = [&](size_t bytes) { const size_t o = off; off += align256(bytes); return o; };
        pl->T = T;
        pl->workers = 0;
        pl->dlast = take(4 * (size_t)G * mdp_stride(s) * nJ);
        pl->tmin = take(4 * out * (size_t)near_groups(T));
        pl->tmin1 = take(4 * out * (size_t)(T * (T + 1) / 2));
        pl->ub = pl->lists = off;
        if (nJ > T) {
            pl->ub = take(4 * out * (size_t)T);
            pl->lists = take((size_t)T * nsplit * (size_t)cdiv(nJ, NT) * (16 * NT + 8));
        }
        pl->costs = off;
        if (build) take(panel_tiles(T, nJ) * (kCostTileFloats * sizeof(float) + BJ * sizeof(float2)));
        pl->part = off;
        if (off > scratch) continue;
        if (nJ <= T) return true;  // one panel: no far phase
        const int64_t slots = (int64_t)((scratch - off) / seg) - (int64_t)T * nsplit;
        pl->workers = (int)std::min<int64_t>(slots, nsm);
        if (pl->workers >= std::min(nsm, 2 * nJ) || (T == 1 && pl->workers >= 1)) return true;
    }
    return false;
}

int launch_dp_fast(const Prefix &P, const double *lamp, int G, int s, void *ws, const Layout &Lw, cudaStream_t st,
                   bool exact_s, bool exact_tables, float *costs, bool build_costs, bool test_stall, bool short_parts,
                   size_t chunk_bytes, bool seeded, bool unbounded, bool tables) {
    double *dp64 = wsp<double>(ws, Lw.dp64);
    int32_t *bp = wsp<int32_t>(ws, Lw.bp);
    // small inputs, very large ones and huge counts take the reference kernel
    if (P.p < 2 * BJ || P.p > kMaxFastP || P.d >= (1 << 24) || s < 3 || s - 2 > 112)
        return launch_dp_reference(P, lamp, G, s, dp64, bp, st);
    int dev = 0, nsm = 0;
    ECASQ_CUDA_TRY(cudaGetDevice(&dev));
    ECASQ_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    FastArgs a{};
    a.v = P.v;
    a.N = P.N;
    a.S = P.S;
    a.S2 = P.S2;
    a.p = P.p;
    a.d = P.d;
    a.ps = P.ps;
    a.invd = 1.0f / (float)P.d;  // IEEE division on the host: correctly rounded
    a.sc = a.sc2 = a.isc2 = 1.0;
    if (P.scale32 != 1.0) {
        // values of another order than fp32 costs are fit for (rare, so that the wait does not matter)
        float *vs = wsp<float>(ws, Lw.keys0);  // the sort's buffers are free now
        int *narrow = reinterpret_cast<int *>(wsp<char>(ws, Lw.keys1)), h = 0;
        ECASQ_CUDA_TRY(cudaMemsetAsync(narrow, 0, sizeof(int), st));
        note_launch();
        k_scale_values<<<(unsigned)cdiv(P.p, 256), 256, 0, st>>>(P.v, vs, P.p, sqrt(P.scale32), narrow);
        ECASQ_LAUNCH_CHECK();
        ECASQ_CUDA_TRY(cudaMemcpyAsync(&h, narrow, sizeof(int), cudaMemcpyDeviceToHost, st));
        ECASQ_CUDA_TRY(cudaStreamSynchronize(st));
        // a spread that no factor brings into fp32: the reference kernel, while its time is seconds
        if (h && P.p <= 32768) return launch_dp_reference(P, lamp, G, s, dp64, bp, st);
        if (!h) {
            a.v = vs;
            a.sc2 = P.scale32;
            a.sc = sqrt(a.sc2);
            a.isc2 = 1.0 / a.sc2;
        }
    }
    a.G = G;
    a.s = s;
    // far tasks: all multipliers in one split while their layers' band state fits shared memory
    a.Gc = std::min(G, std::max(1, 32 * kTaskWords / (s - 2)));
    a.nsplit = (int)cdiv(G, a.Gc);
    a.Gc = (int)cdiv(G, a.nsplit);
    a.nJ = (int)cdiv(P.p, BJ);
    FastParams fp;
    band_factors(s, fp);
    for (int g = 0; g < kMaxG; g++) {
        fp.lam64[g] = g < G ? lamp[g] : 0.0;
        fp.lam32[g] = (float)(fp.lam64[g] * a.sc2);
    }
    size_t rows = (size_t)kMaxG * (size_t)(s + 1) * (size_t)table_stride(Lw.d);
    char *base = wsp<char>(ws, Lw.band);
    auto take = [&](size_t bytes) { char *q = base; base += align256(bytes); return q; };
    a.dp32 = wsp<float>(ws, Lw.dp32);
    a.band = reinterpret_cast<uint64_t *>(take(8 * rows));
    a.need = reinterpret_cast<uint8_t *>(take(rows));
    int *flags = reinterpret_cast<int *>(take(flags_bytes(Lw.d)));  // abort, barrier, task count (64 bits)
    FastParams *dprm = reinterpret_cast<FastParams *>(take(sizeof(FastParams)));
    {
        size_t nJd = (size_t)cdiv(Lw.d, BJ);
        a.corner = reinterpret_cast<float *>(take(32 * nJd * (nJd + 1) / 2));
        a.mdp = reinterpret_cast<float *>(take(4 * (size_t)kMaxG * (size_t)mdp_stride(s) * nJd));
    }
    a.list_cnt = reinterpret_cast<int *>(take(4 * 2 * (size_t)(s + 1)));
    a.wide_cnt = reinterpret_cast<int *>(take(4 * (size_t)(s + 1)));
    char *scratch = base;
    a.mcnt = reinterpret_cast<int32_t *>(take(4 * rows));
    a.members = reinterpret_cast<int32_t *>(take(4 * NMEM * rows));
    a.lists = reinterpret_cast<int32_t *>(take(2 * 4 * rows));
    a.wide = reinterpret_cast<int32_t *>(take(4 * (size_t)kMaxG * (size_t)table_stride(Lw.d)));
    a.mdp_stride = mdp_stride(s);
    a.spin_limit = test_stall ? kTestSpinLimit : kSpinLimit;
    a.hold0 = test_stall ? 1 : 0;
    PanelPlan pl;
    if (!plan_panels(scratch_bytes(Lw.d, s), nsm, a.nJ, G, a.Gc, a.nsplit, s, !costs, &pl)) return ECASQ_EWORKSPACE;
    a.T = pl.T;
    a.workers = short_parts ? std::min(pl.workers, 4) : pl.workers;
    a.first_ord = short_parts ? kLastOrd - 2 : 0;
    a.dlast = reinterpret_cast<float *>(scratch + pl.dlast);
    a.tmin = reinterpret_cast<int *>(scratch + pl.tmin);
    a.tmin1 = reinterpret_cast<float *>(scratch + pl.tmin1);
    a.ub = reinterpret_cast<int *>(scratch + pl.ub);
    a.fbits = reinterpret_cast<uint4 *>(scratch + pl.lists);
    a.funion = reinterpret_cast<uint32_t *>(a.fbits + (size_t)a.T * a.nsplit * (size_t)cdiv(a.nJ, NT) * NT);
    a.fweight = reinterpret_cast<int *>(a.funion + (size_t)a.T * a.nsplit * (size_t)cdiv(a.nJ, NT));
    a.part = reinterpret_cast<float *>(scratch + pl.part);
    a.build = costs ? 0 : 1;
    a.seed = (seeded && s == Lw.s) ? seed_rows(ws, Lw) : nullptr;
    a.costs = costs ? costs : reinterpret_cast<float *>(scratch + pl.costs);
    a.tile_base = 0;
    a.J0 = 0;
    a.J1 = a.nJ;
    // tiles the costs buffer holds at once: the whole triangle, one band (streamed) or one panel
    const size_t cap_tiles = !costs ? panel_tiles(a.T, a.nJ)
                             : chunk_bytes ? chunk_bytes / tile_bytes_with_summary()
                                           : (size_t)cdiv(Lw.d, BJ) * (size_t)(cdiv(Lw.d, BJ) + 1) / 2;
    a.tsum = reinterpret_cast<float2 *>(const_cast<float *>(a.costs) + cap_tiles * kCostTileFloats);
    if (chunk_bytes && cap_tiles < (size_t)a.nJ) return ECASQ_EWORKSPACE;  // one column of tiles must fit
    a.prm = dprm;
    a.abort_flag = flags;
    a.gbar = flags + 1;
    a.work = reinterpret_cast<unsigned long long *>(flags + 2);
    a.st = wsp<DevStatus>(ws, Lw.status);
    float *wf = wsp<float>(ws, Lw.keys1);  // the sort's ping-pong buffer is free now
    a.wf = wf;
    size_t n = (size_t)G * (size_t)(s + 1) * (size_t)P.ps;
    note_launch();
    k_store_params<<<1, 256, 0, st>>>(fp, dprm);
    note_launch();
    k_fast_clear<<<4096, 256, 0, st>>>(dp64, bp, a.dp32, n);
    note_launch();
    k_weights_f32<<<(unsigned)cdiv(P.p, 256), 256, 0, st>>>(P.w, wf, P.p);
    ECASQ_LAUNCH_CHECK();
    ECASQ_CUDA_TRY(cudaMemsetAsync(flags, 0, 4 * sizeof(int), st));
    note_launch();
    // (a warp a block: its binary64 sequence is 5 us of an SM's pipe)
    k_fast_base<<<(unsigned)cdiv(P.p - 1, 32), 32, 0, st>>>(P, a, dp64, bp);
    ECASQ_LAUNCH_CHECK();
    // corner states: needed by every tile that is built (per pass, or once into the table)
    if (a.nJ > 1 && (!costs || build_costs)) {
        note_launch();
        k_corners<<<(unsigned)std::min<int64_t>(cdiv((int64_t)a.nJ * (a.nJ - 1) / 2, 128), (int64_t)nsm * 64), 128, 0, st>>>(a);
        ECASQ_LAUNCH_CHECK();
    }
    int smem_max = 0;
    ECASQ_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    // far tile buffers with room for tcap tasks each, next to the band state and the
    // partial minima
    const size_t nt = (size_t)a.Gc * (s - 2), state = 4 * (2 * nt * BJ + 2 * kBatch * 8 * BJ);
    const size_t fixed = kSmemHead + state + 4 * (size_t)kFarBufs * kCostTileFloats, per = 4 * (size_t)kFarBufs * BK;
    if (fixed + 16 * per > (size_t)smem_max) return ECASQ_ECUDA;
    a.tcap = (int)std::min<size_t>(64, std::max<size_t>(16, std::min(nt, ((size_t)smem_max - fixed) / per)));
    size_t area = std::max(fixed - kSmemHead + a.tcap * per,
                           sizeof(float) * (kNearTiles * kCostTileFloats + (MAXCONS / 32) * 2 * BK +
                                            kNearMults * 2 * kNearTiles * BJ));
    if (a.build) area = std::max(area, kBuildGroups * sizeof(BuildSmem));
    // one stage buffer where two do not fit (8 multipliers: s >= 80).  Such codebooks once went without the skip test: a search
    // at d = 30000, s = 114 with a table took 503 ms (441 with whole column blocks), and takes 206.
    auto stage = [&](int n) { return (n * stage_floats(G, a.mdp_stride) + nt * BJ) * sizeof(float); };
    a.nstage = kSmemHead + stage(2) <= (size_t)smem_max ? 2 : 1;
    area = std::max(area, stage(a.nstage));
    a.bound = a.nJ > a.T ? 1 : 0;
    a.bound_step = unbounded ? 32 : 4;
    const size_t smem = kSmemHead + area;
    // the same limit in every call: another thread's call of another shape may lie between this and the launch
    ECASQ_CUDA_TRY(cudaFuncSetAttribute(k_wavefront, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    int per_sm = 0;
    if (costs && build_costs)
        ECASQ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_build_costs, NPROD, 0));
    // one band of column blocks per round: [J0, J1) whose tiles fit the buffer (all of them
    // when the buffer holds the whole triangle); with streamed costs every band's tiles are
    // built just before its wavefront, else the table is built once per call.  The
    // timer covers the min-plus kernel; with streamed costs, every band's build and
    // wavefront together (the builds are then part of every pass)
    if (chunk_bytes) timer_begin(st);
    for (int J0 = 0; J0 < a.nJ;) {
        int J1 = a.nJ;
        if (chunk_bytes) {
            J1 = J0 + 1;
            const size_t T0 = (size_t)J0 * (J0 + 1) / 2;
            while (J1 < a.nJ && (size_t)(J1 + 1) * (J1 + 2) / 2 - T0 <= cap_tiles) J1++;
        }
        a.J0 = J0;
        a.J1 = J1;
        a.tile_base = chunk_bytes ? (size_t)J0 * (J0 + 1) / 2 : 0;
        if (costs && build_costs) {
            const int64_t ntiles = (int64_t)J1 * (J1 + 1) / 2 - (int64_t)a.tile_base;
            note_launch();
            k_build_costs<<<(unsigned)std::min<int64_t>(ntiles, (int64_t)nsm * std::max(per_sm, 1)), NPROD, 0, st>>>(a);
            ECASQ_LAUNCH_CHECK();
        }
        if (J0 > 0) ECASQ_CUDA_TRY(cudaMemsetAsync(a.gbar, 0, sizeof(int), st));
        // no near minimum carries the first panel's tag (sign 0) yet
        ECASQ_CUDA_TRY(cudaMemsetAsync(a.tmin, 0xFF, 4 * (size_t)near_groups(a.T) * G * (s - 2) * BJ, st));
        if (a.bound) ECASQ_CUDA_TRY(cudaMemsetAsync(a.ub, kNoBound & 0xFF, 4 * (size_t)a.T * G * (s - 2) * BJ, st));
        // one panel: as many CTAs as have near items, or tiles to build
        const int items = near_groups(a.nJ) * (int)cdiv(G, kNearMults);
        const int grid = a.nJ > a.T ? nsm : std::max(items, a.build ? std::min(nsm, a.nJ * (a.nJ + 1) / 2) : 0);
        if (!chunk_bytes) timer_begin(st);
        note_launch();
        void *args[] = {&a};
        ECASQ_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_wavefront, dim3(grid), dim3(MAXCONS), args, smem, st));
        if (!chunk_bytes) timer_end(st);
        ECASQ_LAUNCH_CHECK();
        J0 = J1;
    }
    if (chunk_bytes) timer_end(st);
    // a streamed band or a panel holds only its own tiles: the need and exact stages re-derive
    // the costs they read (any evaluation within the certified bound will do)
    if (chunk_bytes || !costs) {
        a.costs = nullptr;
        a.tile_base = 0;
    }
    const int ilo = exact_s ? s : 2;
    note_launch();
    k_need_init<<<(unsigned)std::min<int64_t>(cdiv((int64_t)G * (s + 1) * P.ps, 256), (int64_t)nsm * 32), 256, 0, st>>>(
        a, ilo, exact_tables ? kNeedAll : tables ? kNeedFinal : kNeedLeast);
    ECASQ_LAUNCH_CHECK();
    ECASQ_CUDA_TRY(cudaMemsetAsync(a.list_cnt, 0, sizeof(int) * 2 * (size_t)(s + 1), st));
    ECASQ_CUDA_TRY(cudaMemsetAsync(a.wide_cnt, 0, sizeof(int) * (size_t)(s + 1), st));
    const unsigned gl = (unsigned)std::min<int64_t>(cdiv((int64_t)G * P.p, 128), (int64_t)nsm * 64);
    for (int i = s; i >= 3; i--) {
        if (exact_tables || tables) {
            note_launch();
            k_need_layer<<<gl, 128, 0, st>>>(a, i);
            ECASQ_LAUNCH_CHECK();
            note_launch();
            k_need_wide<false><<<(unsigned)nsm * 16, 128, 0, st>>>(a, i);
        } else {
            note_launch();
            k_need_wide<true><<<(unsigned)nsm * 16, 128, 0, st>>>(a, i);
        }
        ECASQ_LAUNCH_CHECK();
    }
    note_launch();
    k_fill_unneeded<<<(unsigned)std::min<int64_t>(cdiv((int64_t)G * (s + 1) * P.ps, 256), (int64_t)nsm * 32), 256, 0,
                      st>>>(a, dp64, bp);
    ECASQ_LAUNCH_CHECK();
    for (int i = 3; i <= s; i++) {
        note_launch();
        k_exact_layer<<<(unsigned)nsm * (kExactBlocks + kExactBigBlocks), 128, 0, st>>>(P, a, i, dp64, bp);
        ECASQ_LAUNCH_CHECK();
    }
    return ECASQ_OK;
}

}  // namespace ecasq
