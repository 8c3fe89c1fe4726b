// Judge of the learned normal (internal; the estimator has no counterpart
// in the paper): the residual of a normal on its 3x3x3 stencil and the
// choice between the network's normal and MYC's.
#pragma once

#include <math.h>
#include <stdint.h>

#include "plic.cuh"

namespace vof {

// L1-normalised copy of a normal; false for a zero or non-finite one.
__device__ __forceinline__ bool l1_normalise(const float n[3], float m[3]) {
    const float l1 = fabsf(n[0]) + fabsf(n[1]) + fabsf(n[2]);
    if (!(l1 > 0.f) || !isfinite(l1)) return false;
    m[0] = n[0] / l1;
    m[1] = n[1] / l1;
    m[2] = n[2] / l1;
    return true;
}

// Residual of an L1-normalised normal m on a stencil: the plane of normal m
// holding the centre cell's volume fraction, extended over the 3x3x3 block;
// the mean over the 27 cells of |predicted - actual| fraction, with that
// plane's constant (FP32).  The reflection and ordering of the normal
// and the constants of its volume are taken once per stencil; every cell
// then takes the piecewise closed form (vol_pw_clamped, which gives 0 or 1
// for a cell the plane leaves whole) in one branch-free pass -- a first pass
// that settled the whole cells by a compare and a loop over the cut ones
// cost 27% more instructions, the loop running to the largest cut count of
// the warp.  The value of cell q is st[q * STRIDE] (STRIDE > 1: a
// column of a shared-memory tile).
//
// The arithmetic runs on pairs of cells with the packed FP32 operations of
// this architecture (fma.rn.f32x2 and its kin: two results per issue slot;
// minima, compares and selects stay one by one): the judge is bound by issue.
// Every fused product-sum is written out, so that the compiler's choice of
// contractions cannot move a decision.
struct Residual {
    float e;      // mean |predicted - actual| over the 27 cells
    float alpha;  // the plane constant
};
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 max0(float2 v) { return make_float2(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f)); }
// vol_pw_clamped on two plane constants.
struct VolPW2 {
    float2 S, nab, k_lin, i6abc, ni6abc, i6bc, na, nb, nc, aa;
    float a, x_lin;
    __device__ __forceinline__ explicit VolPW2(const VolPW& p)
        : S(both(p.S)), nab(both(-p.ab)), k_lin(both(p.k_lin)), i6abc(both(p.i6abc)), ni6abc(both(-p.i6abc)),
          i6bc(both(p.i6bc)), na(both(-p.a)), nb(both(-p.b)), nc(both(-p.c)), aa(both(p.a * p.a)),
          a(p.a), x_lin(p.x_lin) {}
    __device__ __forceinline__ float2 operator()(float2 alpha) const {
        const float2 neg = both(-1.f);
        const float2 d = __ffma2_rn(alpha, neg, S);  // S - alpha
        const float2 x = max0(make_float2(fminf(alpha.x, d.x), fminf(alpha.y, d.y)));
        const float2 lin = __fmul2_rn(__ffma2_rn(both(2.f), x, nab), k_lin);
        const float2 v1 = __fmul2_rn(__fmul2_rn(__fmul2_rn(x, x), x), i6abc);
        const float2 tb = max0(__fadd2_rn(x, nb)), tc = max0(__fadd2_rn(x, nc));
        const float2 t = __ffma2_rn(__fmul2_rn(tb, tb), tb, __fmul2_rn(__fmul2_rn(tc, tc), tc));
        const float2 q = __ffma2_rn(__fmul2_rn(both(3.f), x), __fadd2_rn(x, na), aa);
        const float2 v3 = __ffma2_rn(q, i6bc, __fmul2_rn(t, ni6abc));
        const float2 v = make_float2(x.x > x_lin ? lin.x : (x.x <= a ? v1.x : v3.x),
                                     x.y > x_lin ? lin.y : (x.y <= a ? v1.y : v3.y));
        const float2 w = __ffma2_rn(v, neg, both(1.f));  // 1 - v
        return make_float2(d.x < alpha.x ? w.x : v.x, d.y < alpha.y ? w.y : v.y);
    }
};
template <int STRIDE>
static __device__ __noinline__ Residual normal_residual_m(const float* st, float m0, float m1, float m2) {
    // x_i -> 1 - x_i for a negative component moves the constant by |m_i|
    const float off = fmaxf(-m0, 0.f) + fmaxf(-m1, 0.f) + fmaxf(-m2, 0.f);
    float a = fabsf(m0), b = fabsf(m1), c = fabsf(m2);
    sort3(a, b, c);
    const VolPW p = vol_pw_make(a, b, c);
    // the plane constant in the reflected frame, and in the grid's
    const float A = alpha_pw(p, st[13 * STRIDE]);
    const VolPW2 vol(p);
    float e = 0.f;
    // one rolled loop over the three planes along z keeps the code small
    // enough for the instruction cache; each plane's 9 cells are unrolled
#pragma unroll 1
    for (int k = -1; k <= 1; ++k) {
        const float* sk = st + (k + 1) * 9 * STRIDE;
        const float2 mk = both(m2 * (float)k);
#pragma unroll
        for (int q = 0; q < 9; q += 2) {
            const int r = q < 8 ? q + 1 : q;  // the ninth cell stands twice
            const float2 s = make_float2(__fadd_rn(m0 * (float)(q % 3 - 1), m1 * (float)(q / 3 - 1)),
                                         __fadd_rn(m0 * (float)(r % 3 - 1), m1 * (float)(r / 3 - 1)));
            const float2 v = vol(__ffma2_rn(__fadd2_rn(s, mk), both(-1.f), both(A)));
            e += fabsf(v.x - sk[q * STRIDE]);
            if (q < 8) e += fabsf(v.y - sk[r * STRIDE]);
        }
    }
    return {e * (1.f / 27.f), A - off};
}

// Residual of any normal n (+inf for a zero or non-finite one).
__device__ __forceinline__ float normal_residual(const float st[27], const float n[3]) {
    float m[3];
    if (!l1_normalise(n, m)) return INFINITY;
    return normal_residual_m<1>(st, m[0], m[1], m[2]).e;
}

// The learned normal as the step uses it: the network's normal nn (original
// frame, L1-normalised by division) is kept when the residual of its plane
// is at most tol, or no larger than that of MYC's normal; otherwise MYC's.
// m gets the choice; returns true when the network's was kept.
__device__ __forceinline__ bool judged_normal(const float st[27], const float nn[3], float tol, float m[3]) {
    float mn[3];
    const float e_net = l1_normalise(nn, mn) ? normal_residual_m<1>(st, mn[0], mn[1], mn[2]).e : INFINITY;
    bool keep = e_net <= tol;
    if (!keep) {
        myc_normal(st, m);
        keep = e_net <= normal_residual_m<1>(st, m[0], m[1], m[2]).e;
    }
    if (keep) {
        m[0] = mn[0];
        m[1] = mn[1];
        m[2] = mn[2];
    }
    return keep;
}

}  // namespace vof
