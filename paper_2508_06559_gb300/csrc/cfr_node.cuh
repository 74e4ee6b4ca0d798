// The arithmetic of one (active node, score slot) of a CFR iteration, shared by every sweep (one
// block per item, thread-block clusters, level streaming), so that their results are the same bit
// for bit.
#pragma once

#include "pasur_internal.cuh"

namespace pasur {

// Pairwise sum of D values (a short dependency chain: about log2(D) additions deep).
template <int D>
__device__ __forceinline__ float tree_sum(const float *x) {
    if (D == 1) return x[0];
    if (D == 2) return x[0] + x[1];
    constexpr int H = D / 2;
    return tree_sum<H>(x) + tree_sum<D - H>(x + H);
}

// 1 / s for a positive regret sum: the fast reciprocal (at most 2 ulp; the sum is a normal
// number, since counted regrets exceed the dead zone).
__device__ __forceinline__ float rcp_pos(float s) { return __fdividef(1.f, s); }

// Regret matching over the regrets r of D > 1 child edges: the children's reaches own * sigma.
template <int D>
__device__ __forceinline__ void rm_reach(const float *r, float own, float thr, float *x) {
    float rp[D];
#pragma unroll
    for (int a = 0; a < D; a++) rp[a] = r[a] > thr ? r[a] : 0.f;
    const float sum = tree_sum<D>(rp);
    const bool pos = sum > 0.f;
    // pos: rp * scale (an fma with a zero addend rounds the product alone); otherwise every rp is
    // zero and the fma gives the uniform share: one instruction per child instead of two
    const float scale = pos ? own * rcp_pos(sum) : 0.f, u = pos ? 0.f : own * (1.f / (float)D);
#pragma unroll
    for (int a = 0; a < D; a++) x[a] = __fmaf_rn(rp[a], scale, u);
}

// Value of a node from the regrets r, strategy sums s and values v of its D child edges, then
// R(h,a) += s_p pi_{-p}(h) (v(h.a) - v(h)) and S(h,a) += pi_p(h) sigma(h,a) in place in r and s.
// Returns v(h).
template <int VARIANT, int D>
__device__ __forceinline__ float bu_vals(float *r, const float *v, float *s, float pp, float spo, float thr, float fpos,
                                         float fneg, float fs) {
    float rp[D];
#pragma unroll
    for (int a = 0; a < D; a++) rp[a] = r[a] > thr ? r[a] : 0.f;
    const float sum = tree_sum<D>(rp);
    const bool pos = sum > 0.f;
    const float inv = pos ? rcp_pos(sum) : 0.f, u = pos ? 0.f : 1.f / (float)D;
    float sg[D], dv[D];
#pragma unroll
    for (int a = 0; a < D; a++) {
        sg[a] = __fmaf_rn(rp[a], inv, u);  // rp * inv, or the uniform share (as in td_node)
        dv[a] = a == 0 ? 0.f : sg[a] * (v[a] - v[0]);
    }
    const float vh = D == 1 ? v[0] : v[0] + tree_sum<D>(dv);
#pragma unroll
    for (int a = 0; a < D; a++) {
        const float inst = spo * (v[a] - vh);
        if (VARIANT == 1) {
            r[a] = r[a] * (r[a] > 0.f ? fpos : fneg) + inst;
            s[a] = s[a] * fs + pp * sg[a];
        } else {
            r[a] = r[a] + inst;
            s[a] = s[a] + pp * sg[a];
        }
    }
    return vh;
}

}  // namespace pasur
