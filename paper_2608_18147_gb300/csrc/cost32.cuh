// cost32.cuh -- interval costs in certified fp32 (App. E quantities): compensated recurrences that
// add one point at a time, all terms non-negative, within 24u of the exact cost (u = 2^-24; the
// bound is derived at the head of dp_fast.cu).
#pragma once

#include <algorithm>

#include "common.cuh"

namespace ecasq {

// ------------------------------------------------------------ fp32 numerics

// Sum2 step (Ogita, Rump, Oishi 2005): x + c carries the running sum of
// non-negative terms; TwoSum keeps the rounding error of each addition.
__device__ __forceinline__ void comp_add(float &x, float &c, float t) {
    float s = __fadd_rn(x, t);
    float bb = __fsub_rn(s, x);
    float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(t, bb));
    x = s;
    c = __fadd_rn(c, e);
}

// Reciprocal from rcp.approx plus one Newton step: relative error <= u/2 + 2^-46
// (no slow-path branch, unlike the IEEE-rounded intrinsic).
__device__ __forceinline__ float rcp_nr(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    float e = __fmaf_rn(-x, r, 1.0f);
    return __fmaf_rn(r, e, r);
}

// -log2(1 - z) for z in [0, 1/2], from log(1 - z) = -2 atanh(z / (2 - z)).
__device__ __forceinline__ float neg_log2_1m(float z) {
    float t = __fmul_rn(z, rcp_nr(__fsub_rn(2.0f, z)));  // t in [0, 1/3]
    float t2 = __fmul_rn(t, t);
    // 2 (t + t^3/3 + ... + t^15/15) / ln 2; the next term is below 2^-26 t
    float q = 1.0f / 15.0f;
    q = __fmaf_rn(q, t2, 1.0f / 13.0f);
    q = __fmaf_rn(q, t2, 1.0f / 11.0f);
    q = __fmaf_rn(q, t2, 1.0f / 9.0f);
    q = __fmaf_rn(q, t2, 1.0f / 7.0f);
    q = __fmaf_rn(q, t2, 1.0f / 5.0f);
    q = __fmaf_rn(q, t2, 1.0f / 3.0f);
    q = __fmaf_rn(q, t2, 1.0f);
    return __fmul_rn(__fmul_rn(t, q), 2.8853900817779268f);  // 2 / ln 2
}

// h(y) = -y log2 y for y in [0, 1/2] (y = 0 gives 0), without branches.
__device__ __forceinline__ float h32_small(float y) {
    float r = __fmul_rn(y, -__log2f(fmaxf(y, 1e-37f)));
    return (y > 0.0f) ? fmaxf(r, 0.0f) : 0.0f;
}
// h(y) for y in [0, 1], `comp` = 1 - y computed from the complementary mass.  The
// series for y > 1/2 is a branch: only intervals holding more than half of all entries
// reach it, and a warp whose lanes have none skips it.
__device__ __forceinline__ float h32_any(float y, float comp) {
    float l = -__log2f(fmaxf(y, 1e-37f));
    if (y > 0.5f) l = neg_log2_1m(fminf(fmaxf(comp, 0.0f), 0.5f));
    float r = __fmul_rn(y, l);
    return (y > 0.0f) ? fmaxf(r, 0.0f) : 0.0f;
}

// Recurrence state of one column j while k descends: N = sum w, E = sum w (v_j - v_t),
// A = sum w (v_t - v_k), C = sum w (v_j - v_t)(v_t - v_k) over t in (k, j].
struct Rec {
    float N, E, Ec, A, Ac, C, Cc;
};

// Interval cost of (k, j) from the state: C and Phi = h(U/d) + h(D/d) (Sec. 5).
// At most one of U, D exceeds d/2 (U + D <= d), so only the larger mass needs
// the 1 - y form.
__device__ __forceinline__ void rec_emit(const Rec &r, float vj, float vk, float d_f, float invd, float &Cout,
                                         float &Phi) {
    float Eu = __fadd_rn(r.E, r.Ec), Au = __fadd_rn(r.A, r.Ac);
    Cout = __fadd_rn(fmaxf(__fadd_rn(r.C, r.Cc), 0.0f), 0.0f);  // >= +0 (no -0)
    float L = __fsub_rn(vj, vk);
    float rL = rcp_nr(L);
    float D = __fmul_rn(Eu, rL), U = __fmul_rn(Au, rL);
    float mbig = fmaxf(U, D), msmall = fminf(U, D);
    float out = __fsub_rn(d_f, r.N);  // mass outside the interval (exact)
    float comp = __fmul_rn(__fadd_rn(out, msmall), invd);
    Phi = __fadd_rn(__fadd_rn(h32_small(__fmul_rn(msmall, invd)), h32_any(__fmul_rn(mbig, invd), comp)), 0.0f);
}

// Add point t = k+1 (moving from k+1 to k): vt = v_{k+1}, wt = w_{k+1}, dk = v_{k+1} - v_k.
__device__ __forceinline__ void rec_step(Rec &r, float vj, float vt, float wt, float dk) {
    r.N = __fadd_rn(r.N, wt);
    comp_add(r.E, r.Ec, __fmul_rn(wt, __fsub_rn(vj, vt)));
    float Eu = __fadd_rn(r.E, r.Ec);
    comp_add(r.A, r.Ac, __fmul_rn(dk, r.N));
    comp_add(r.C, r.Cc, __fmul_rn(dk, Eu));
}

__device__ __forceinline__ Rec rec_empty() { return {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}; }

// Certified band factors of the fp32 recurrence: eps_2 = 1.0001u, eps_i = max(eps_{i-1}, 24u) + 1.0001u;
// tau_i >= 2 eps_i / (1 - eps_i), with margin.
inline void band_factors(int s, float *tau, float *eps_out) {
    const double u = 1.0 / 16777216.0;
    for (int i = 0; i <= kMaxS; i++) tau[i] = eps_out[i] = 0.f;
    double eps = 1.0001 * u;
    eps_out[2] = (float)eps;
    for (int i = 3; i <= s; i++) {
        eps = std::max(eps, 24.0 * u) + 1.0001 * u;
        eps_out[i] = (float)eps;
        tau[i] = (float)(2.0 * eps / (1.0 - eps) * 1.001 + 2.0 * u);
    }
}

}  // namespace ecasq
