// PLIC geometry in double for GB300, whose FP64 rate is 1/64 of its FP32 rate
// (a warp's FP64 instruction holds its scheduler's FP64 unit for 64 cycles):
// the bound of every FP64 reconstruction is the number of FP64 instructions,
// so the forms below are chosen for few of them.
//
//   * Compares of non-negative values run on their bit patterns (integer ALU).
//   * Nothing is normalised: the plane constant and the volume are homogeneous
//     in the normal, so a face flux needs no division by |m|_1.
//   * The volume takes one division: inclusion-exclusion over the vertices
//     (Scardovelli & Zaleski 2000, JCP 164) with its terms paired so that no
//     large term is divided by a small product (see vol_pw in plic.cuh).
//   * The plane constant's cubic regions start from the FP32 closed form in
//     variables scaled by the middle component (all of order one) and take
//     two FP64 Newton steps whose slope is a float: the seed's relative error
//     e0 < 1e-6 becomes e0^2 + 1e-7 e0 ~ 1e-13 after the first step and
//     1e-7 of that after the second, below one ulp.
//
// Every product-sum is an explicit fma(), so that units compiled with and
// without contraction give the same bits.
//
// Against quadruple precision on a million random planes, fractions and
// Courant numbers (tiny and zero components included): flux within 4.6e-16
// (mean 1.17e-17), plane constant within 3.1e-16 (mean 3.4e-17); the
// piecewise Gauss evaluation and its Newton inversion that stood here before
// gave 5.6e-16 (1.37e-17) and 3.6e-16 (4.2e-17).  Times: k_face_flux_bx.
#pragma once

#include <math.h>
#include <stdint.h>

namespace vof {

#ifdef __CUDACC__
#define VOF_HD __host__ __device__ __forceinline__
#else
#define VOF_HD static inline
#endif

VOF_HD long long bits64(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    long long b;
    __builtin_memcpy(&b, &v, 8);
    return b;
#endif
}
VOF_HD double from_bits64(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double v;
    __builtin_memcpy(&v, &b, 8);
    return v;
#endif
}
VOF_HD double abs64(double v) { return from_bits64(bits64(v) & 0x7fffffffffffffffLL); }
VOF_HD bool negative64(double v) { return bits64(v) < 0; }
// p < q, p <= q for non-negative p and q (no NaN), on the integer ALU.
VOF_HD bool lt_pos(double p, double q) { return bits64(p) < bits64(q); }
VOF_HD bool le_pos(double p, double q) { return bits64(p) <= bits64(q); }
// max(v, 0) for any v (-0 gives +0).
VOF_HD double plus64(double v) { return bits64(v) < 0 ? 0.0 : v; }

VOF_HD void sort3_pos(double& a, double& b, double& c) {
    double t;
    if (lt_pos(b, a)) { t = a; a = b; b = t; }
    if (lt_pos(c, b)) { t = b; b = c; c = t; }
    if (lt_pos(b, a)) { t = a; a = b; b = t; }
}

// Cube root of t >= 0: FP32 root of the mantissa (exponent a multiple of
// three), two Newton steps in double with a float slope.
VOF_HD double cbrt64(double t) {
    if (lt_pos(t, 1e-300)) return 0.0;
    const int e = (int)(bits64(t) >> 52) - 1023;          // >= -997
    const int k = (e + 1200) / 3 - 400;                   // floor(e / 3)
    const double m = t * from_bits64((long long)(1023 - 3 * k) << 52);  // in [1, 8)
    const float yf = cbrtf((float)m);
    const double r = (double)(1.f / (3.f * yf * yf));
    double y = (double)yf;
    y = fma(-fma(y * y, y, -m), r, y);
    y = fma(-fma(y * y, y, -m), r, y);
    return y * from_bits64((long long)(1023 + k) << 52);
}

// Volume under the plane a x + b y + c z < x in the unit cube, sorted
// 0 <= a <= b <= c, c > 0, 0 <= x <= (a + b + c) / 2.
VOF_HD double vol64_half(double a, double b, double c, double x) {
    double num, den;
    if (le_pos(x, a)) {
        num = x * x * x;
        den = 6.0 * a * b * c;
    } else if (lt_pos(a + b, x)) {  // the prism (x <= S/2 leaves it to c > a + b)
        num = fma(2.0, x, -(a + b));
        den = 2.0 * c;
    } else {
        const double q = fma(3.0 * x, x - a, a * a);
        const double tb = x - b;
        den = 6.0 * b * c;
        num = q;
        if (bits64(tb) > 0) {  // not at x = b, where a may be zero
            const double tc = plus64(x - c);
            num = fma(a, q, -fma(tb * tb, tb, tc * tc * tc));
            den *= a;
        }
    }
    // a divisor this small belongs to a plane whose volume is below 1e-90
    return lt_pos(den, 1e-290) ? 0.0 : num / den;
}

// The same for any x; S = a + b + c > 0.
VOF_HD double vol64(double a, double b, double c, double x) {
    const double S = a + b + c, y = S - x;
    if (bits64(x) <= 0) return 0.0;
    if (bits64(y) <= 0) return 1.0;
    if (lt_pos(y, x)) return 1.0 - vol64_half(a, b, c, y);
    return vol64_half(a, b, c, x);
}

// Root x in (0, S/2] of vol64_half(a, b, c, x) = v, 0 < v <= 1/2, sorted
// 0 <= a <= b <= c, c > 0.  In units of b (p = a/b, w = c v / b, g = c/b):
//   6w <= p^2:            x^3 = 6 p w
//   6w <= 3 - 3p + p^2:   3x(x - p) + p^2 = 6w
//   c >= a + b, 2w >= 1 + p:  the prism, x = w + (1 + p)/2
//   else  p (3x(x - p) + p^2 - 6w) = (x - 1)^3 + (x - g)_+^3, seeded by the
//   middle root of the cubic in trigonometric form (alpha_sorted_pw).
VOF_HD double alpha64_half(double a, double b, double c, double v) {
    if (lt_pos(b, 1e-30 * c)) return c * v;  // a plane across one axis (off by < 1e-30 c)
    const double cv = c * v, ib = 1.0 / b;
    const double p = a * ib, w6 = 6.0 * cv * ib, p2 = p * p;
    if (le_pos(w6, p2)) return b * cbrt64(p * w6);
    if (!negative64(fma(3.0, 1.0 - p, p2) - w6))
        return b * (0.5 * (p + sqrt(fma(-1.0 / 3.0, p2, (4.0 / 3.0) * w6))));
    const double ab = a + b;
    const bool prism = le_pos(ab, c);
    if (prism && le_pos(ab, 2.0 * cv)) return fma(0.5, ab, cv);
    const double g = c * ib;
    const double hi = prism ? 1.0 + p : 0.5 * (1.0 + p + g);
    // seed
    const float pf = (float)p, gf = (float)g, wf = (float)w6 * (1.f / 6.f);
    float center, r, z;
    bool last = false;  // beyond x = g
    if (!prism) {
        const float gp = gf - pf, g1 = gf - 1.f;
        last = 6.f * pf * wf > gf * gf * gf - gp * gp * gp - g1 * g1 * g1;
    }
    if (!last) {
        r = sqrtf(2.f * pf);
        center = 1.f + pf;
        z = 3.f * (center - 2.f * wf) / (4.f * r);
    } else {
        const float s = 1.f + pf + gf;
        r = sqrtf(fmaxf(pf + gf + pf * gf - 0.25f * s * s, 0.f));
        center = 0.5f * s;
        z = 0.75f * pf * (gf - 2.f * wf) / (r * r * r);
    }
    z = fminf(fmaxf(z, -1.f), 1.f);
    const float xf = center + 2.f * r * cosf(acosf(z) * (1.f / 3.f) - 2.09439510239f);
    double x = (double)xf;
    if (!(x > 1.0)) x = 1.0;  // also a NaN of a degenerate seed
    if (lt_pos(hi, x)) x = hi;
    if (lt_pos(p, 1e-20)) return b * x;  // the region is narrower than an ulp
    // Newton: G(x) = p (3x(x - p) + p^2 - 6w) - (x - 1)^3 - (x - g)_+^3
    const float xs = (float)x, t1 = xs - 1.f, t2 = fmaxf(xs - gf, 0.f);
    const double rs = (double)(1.f / (pf * (6.f * xs - 3.f * pf) - 3.f * (t1 * t1 + t2 * t2)));
    const double k0 = p2 - w6;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int it = 0; it < 2; ++it) {
        const double tb = x - 1.0, tc = plus64(x - g);
        const double G = fma(p, fma(3.0 * x, x - p, k0), -fma(tb * tb, tb, tc * tc * tc));
        x = fma(-G, rs, x);
    }
    if (lt_pos(hi, x)) x = hi;
    return b * x;
}

// Plane constant of the reflected, sorted normal for a fraction cv in (0, 1).
VOF_HD double alpha64(double a, double b, double c, double cv) {
    const bool flip = lt_pos(0.5, cv);
    const double x = alpha64_half(a, b, c, flip ? 1.0 - cv : cv);
    return flip ? (a + b + c) - x : x;
}

// Mixed-Youngs-Centred direction of a stencil (myc_normal in plic.cuh gives
// the rule), not normalised; returns its L1 norm.  The Youngs sums run
// through partial sums (51 additions instead of 81); the
// centred-column candidates, whose own component is +-1, compare by their L1
// norms instead of three divisions -- the quotients decide only where two
// norms agree to two ulps, so that symmetric stencils keep their choice.
VOF_HD double myc_direction64(const double* st, double m[3]) {
#define VOF_S(i, j, k) st[((k) + 1) * 9 + ((j) + 1) * 3 + ((i) + 1)]
    // Youngs: differences first (exact between close values), then the
    // (1, 2, 1) weights along the two other axes
    auto smooth = [](double lo, double mid, double hi) { return fma(2.0, mid, lo + hi); };
    double y[3];
    {
        double s[3];
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = -1; k <= 1; ++k)
            s[k + 1] = smooth(VOF_S(-1, -1, k) - VOF_S(1, -1, k), VOF_S(-1, 0, k) - VOF_S(1, 0, k),
                              VOF_S(-1, 1, k) - VOF_S(1, 1, k));
        y[0] = smooth(s[0], s[1], s[2]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = -1; k <= 1; ++k)
            s[k + 1] = smooth(VOF_S(-1, -1, k) - VOF_S(-1, 1, k), VOF_S(0, -1, k) - VOF_S(0, 1, k),
                              VOF_S(1, -1, k) - VOF_S(1, 1, k));
        y[1] = smooth(s[0], s[1], s[2]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int j = -1; j <= 1; ++j)
            s[j + 1] = smooth(VOF_S(-1, j, -1) - VOF_S(-1, j, 1), VOF_S(0, j, -1) - VOF_S(0, j, 1),
                              VOF_S(1, j, -1) - VOF_S(1, j, 1));
        y[2] = smooth(s[0], s[1], s[2]);
    }
    // centred columns: (b, c) components of the candidate along each axis
    const double cx_b = (((VOF_S(-1, -1, 0) + VOF_S(0, -1, 0)) + VOF_S(1, -1, 0)) -
                         ((VOF_S(-1, 1, 0) + VOF_S(0, 1, 0)) + VOF_S(1, 1, 0))) * 0.5;
    const double cx_c = (((VOF_S(-1, 0, -1) + VOF_S(0, 0, -1)) + VOF_S(1, 0, -1)) -
                         ((VOF_S(-1, 0, 1) + VOF_S(0, 0, 1)) + VOF_S(1, 0, 1))) * 0.5;
    const double cy_b = (((VOF_S(-1, -1, 0) + VOF_S(-1, 0, 0)) + VOF_S(-1, 1, 0)) -
                         ((VOF_S(1, -1, 0) + VOF_S(1, 0, 0)) + VOF_S(1, 1, 0))) * 0.5;
    const double cy_c = (((VOF_S(0, -1, -1) + VOF_S(0, 0, -1)) + VOF_S(0, 1, -1)) -
                         ((VOF_S(0, -1, 1) + VOF_S(0, 0, 1)) + VOF_S(0, 1, 1))) * 0.5;
    const double cz_b = (((VOF_S(-1, 0, -1) + VOF_S(-1, 0, 0)) + VOF_S(-1, 0, 1)) -
                         ((VOF_S(1, 0, -1) + VOF_S(1, 0, 0)) + VOF_S(1, 0, 1))) * 0.5;
    const double cz_c = (((VOF_S(0, -1, -1) + VOF_S(0, -1, 0)) + VOF_S(0, -1, 1)) -
                         ((VOF_S(0, 1, -1) + VOF_S(0, 1, 0)) + VOF_S(0, 1, 1))) * 0.5;
#undef VOF_S
    // L1 norms, summed in component order
    const double lx = (1.0 + abs64(cx_b)) + abs64(cx_c);
    const double ly = (abs64(cy_b) + 1.0) + abs64(cy_c);
    const double lz = (abs64(cz_b) + abs64(cz_c)) + 1.0;
    auto better = [](double l, double best) {  // 1/l > 1/best as rounded quotients
        const long long dl = bits64(best) - bits64(l);
        if (dl > 2) return true;
        if (dl <= 0) return false;
        return 1.0 / l > 1.0 / best;
    };
    double lbest = lx;
    m[0] = negative64(y[0]) ? -1.0 : 1.0;
    m[1] = cx_b;
    m[2] = cx_c;
    if (better(ly, lbest)) {
        lbest = ly;
        m[0] = cy_b;
        m[1] = negative64(y[1]) ? -1.0 : 1.0;
        m[2] = cy_c;
    }
    if (better(lz, lbest)) {
        lbest = lz;
        m[0] = cz_b;
        m[1] = cz_c;
        m[2] = negative64(y[2]) ? -1.0 : 1.0;
    }
    const double ax = abs64(y[0]), ay = abs64(y[1]), az = abs64(y[2]);
    const double ny = ax + ay + az;
    double ymax = lt_pos(ax, ay) ? ay : ax;
    ymax = lt_pos(ymax, az) ? az : ymax;
    // Youngs where ymax / ny < 1 / lbest (the quotients near a tie)
    bool youngs = false;
    if (le_pos(1e-30, ny)) {
        const double t = ymax * lbest;
        const long long dl = bits64(ny) - bits64(t);
        youngs = dl > 4 || (dl >= -4 && ymax / ny < 1.0 / lbest);
    }
    if (youngs) {
        m[0] = y[0];
        m[1] = y[1];
        m[2] = y[2];
        return ny;
    }
    return lbest;
}

// Flux through a face of the donor of fraction cv in (0, 1) with normal
// direction m (any scale); s is the signed Courant number.  In the frame
// reflected to non-negative components the swept slab [1 - s, 1] (s > 0) or
// [0, |s|] (s < 0) keeps or swaps its end with the sign of m_d; it is mapped
// onto the unit cube by n_d -> n_d |s|, alpha -> alpha - n_d x0.
VOF_HD double face_flux64(const double m[3], double cv, int d, double s) {
    double n0 = abs64(m[0]), n1 = abs64(m[1]), n2 = abs64(m[2]);
    double a = n0, b = n1, c = n2;
    sort3_pos(a, b, c);
    const double al = alpha64(a, b, c, cv);
    const double as = abs64(s);
    const double nd = d == 0 ? n0 : (d == 1 ? n1 : n2), md = d == 0 ? m[0] : (d == 1 ? m[1] : m[2]);
    const bool far_end = negative64(s) == negative64(md);
    const double x = far_end ? fma(-nd, 1.0 - as, al) : al;
    const double sd = nd * as;
    if (d == 0) n0 = sd;
    else if (d == 1) n1 = sd;
    else n2 = sd;
    sort3_pos(n0, n1, n2);
    if (!lt_pos(0.0, n2)) return bits64(x) > 0 ? s : 0.0;
    return s * vol64(n0, n1, n2, x);
}

}  // namespace vof
