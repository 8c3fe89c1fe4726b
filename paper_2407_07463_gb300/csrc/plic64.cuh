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
// 0 <= a <= b <= c, c > 0, 0 <= x <= (a + b + c) / 2, by its piece.
enum VolPiece { kVolTip = 0, kVolPrism = 1, kVolEdge = 2, kVolCorner = 3 };
VOF_HD int vol64_piece(double a, double b, double c, double x) {
    if (le_pos(x, a)) return kVolTip;
    if (lt_pos(a + b, x)) return kVolPrism;  // (x <= S/2 leaves it to c > a + b)
    return le_pos(x, b) ? kVolEdge : kVolCorner;
}
VOF_HD double vol64_of(int piece, double a, double b, double c, double x) {
    double num, den;
    if (piece == kVolTip) {
        num = x * x * x;
        den = 6.0 * a * b * c;
    } else if (piece == kVolPrism) {
        num = fma(2.0, x, -(a + b));
        den = 2.0 * c;
    } else {
        num = fma(3.0 * x, x - a, a * a);
        den = 6.0 * b * c;
        if (piece == kVolCorner) {
            const double tb = x - b, tc = plus64(x - c);
            num = fma(a, num, -fma(tb * tb, tb, tc * tc * tc));
            den *= a;
        }
    }
    // a divisor this small belongs to a plane whose volume is below 1e-90
    return lt_pos(den, 1e-290) ? 0.0 : num / den;
}
VOF_HD double vol64_half(double a, double b, double c, double x) {
    return vol64_of(vol64_piece(a, b, c, x), a, b, c, x);
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
enum AlphaPiece { kAlphaLinear = 0, kAlphaCbrt = 1, kAlphaSqrt = 2, kAlphaCubic = 3 };
// 1 / b for b within FP32's range: two Newton steps from the FP32 quotient.
VOF_HD double rcp64(double b) {
    double r = (double)(1.f / (float)b);
    r = fma(fma(-b, r, 1.0), r, r);
    return fma(fma(-b, r, 1.0), r, r);
}
// The piece the root lies in and its scaled variables p, w6 = 6w and g (g only
// for the cubic); the linear pieces' root in x.  c within 2^-20 .. 2^20.
VOF_HD int alpha64_piece(double a, double b, double c, double v, double& p, double& w6, double& g, double& x) {
    const double cv = c * v;
    x = cv;
    if (lt_pos(b, 1e-30 * c)) return kAlphaLinear;  // a plane across one axis (off by < 1e-30 c)
    const double ib = rcp64(b);
    p = a * ib;
    w6 = 6.0 * cv * ib;
    const double p2 = p * p;
    if (le_pos(w6, p2)) return kAlphaCbrt;
    if (!negative64(fma(3.0, 1.0 - p, p2) - w6)) return kAlphaSqrt;
    const double ab = a + b;
    if (le_pos(ab, c) && le_pos(ab, 2.0 * cv)) {
        x = fma(0.5, ab, cv);
        return kAlphaLinear;
    }
    g = c * ib;
    return kAlphaCubic;
}
VOF_HD double alpha64_cbrt(double p, double w6, double b) { return b * cbrt64(p * w6); }
VOF_HD double alpha64_sqrt(double p, double w6, double b) {
    return b * (0.5 * (p + sqrt(fma(-1.0 / 3.0, p * p, (4.0 / 3.0) * w6))));
}
VOF_HD double alpha64_cubic(double p, double w6, double g, double b) {
    // seed
    const float pf = (float)p, gf = (float)g, wf = (float)w6 * (1.f / 6.f);
    const double p1 = 1.0 + p;
    const bool prism = le_pos(p1, g);
    const double hi = prism ? p1 : 0.5 * (p1 + g);
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
    double x = xf > 1.f ? (double)xf : 1.0;  // (1 also for a NaN of a degenerate seed)
    if (lt_pos(hi, x)) x = hi;
    if (lt_pos(p, 1e-20)) return b * x;  // the region is narrower than an ulp
    // Newton: G(x) = p (3x(x - p) + p^2 - 6w) - (x - 1)^3 - (x - g)_+^3
    const float xs = (float)x, t1 = xs - 1.f, t2 = fmaxf(xs - gf, 0.f);
    const double rs = (double)(1.f / (pf * (6.f * xs - 3.f * pf) - 3.f * (t1 * t1 + t2 * t2)));
    const double k0 = fma(p, p, -w6);
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
VOF_HD double alpha64_half(double a, double b, double c, double v) {
    double p, w6, g, x;
    const int piece = alpha64_piece(a, b, c, v, p, w6, g, x);
    if (piece == kAlphaCbrt) return alpha64_cbrt(p, w6, b);
    if (piece == kAlphaSqrt) return alpha64_sqrt(p, w6, b);
    if (piece == kAlphaCubic) return alpha64_cubic(p, w6, g, b);
    return x;
}

// Plane constant of the reflected, sorted normal for a fraction cv in (0, 1).
VOF_HD double alpha64(double a, double b, double c, double cv) {
    const bool flip = lt_pos(0.5, cv);
    const double x = alpha64_half(a, b, c, flip ? 1.0 - cv : cv);
    return flip ? (a + b + c) - x : x;
}

// A double as a whole number of 2^(eref - 1080), eref >= its biased exponent
// (bits below that are dropped): |result| < 2^58.
VOF_HD long long fixed64(double v, int eref) {
    const long long b = bits64(v);
    const int e = (int)(b >> 52) & 0x7ff;
    const long long m = ((b & 0xfffffffffffffLL) | 0x10000000000000LL) << 5;
    const int sh = eref - e;
    const long long q = m >> (sh > 62 ? 62 : sh);
    return b < 0 ? -q : q;
}
// A whole number times 2^sh as a double (0 stays 0).
VOF_HD double scaled64(long long n, int sh) {
    const double v = (double)n;
    return n == 0 ? 0.0 : from_bits64(bits64(v) + ((long long)sh << 52));
}
VOF_HD unsigned long long mag64(long long v) { return (unsigned long long)(v < 0 ? -v : v); }

// Mixed-Youngs-Centred direction of a stencil (myc_normal in plic.cuh gives
// the rule), not normalised: its largest component lies in 1 .. 2.  The hundred
// additions run on 64-bit integers (the integer pipes are idle in the FP64
// kernels): the fractions become whole numbers of 2^-57 of the largest
// neighbour's binade, 32 times finer than that value's own last place, so that
// sums and differences are exact and no less accurate than in double.  The
// candidates compare by T, their L1 norm being 1 + T/2, Youngs against the best
// candidate in float; near a tie both take the rounded quotients of the rule in
// double.
VOF_HD void myc_direction64(const double* st, double m[3]) {
#define VOF_S(i, j, k) q[((k) + 1) * 9 + ((j) + 1) * 3 + ((i) + 1)]
    int eref = 600;  // a stencil below 2^-423 counts as empty
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 27; ++c) {
        const int e = (int)(bits64(st[c]) >> 52) & 0x7ff;
        if (c != 13) eref = e > eref ? e : eref;  // (the centre enters no sum)
    }
    if (eref == 0x7ff) {  // an infinity or a NaN beside the cell
        m[0] = m[1] = m[2] = from_bits64(0x7ff8000000000000LL);
        return;
    }
    long long q[27];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 27; ++c) q[c] = c == 13 ? 0 : fixed64(st[c], eref);
    // Youngs: differences along the axis, weights (1, 2, 1) along the others
    auto smooth = [](long long lo, long long mid, long long hi) { return lo + hi + 2 * mid; };
    long long y[3];
    {
        long long s[3];
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
    // centred columns: twice the (b, c) components of the candidate along each axis
    const long long xb = (VOF_S(-1, -1, 0) + VOF_S(0, -1, 0) + VOF_S(1, -1, 0)) -
                         (VOF_S(-1, 1, 0) + VOF_S(0, 1, 0) + VOF_S(1, 1, 0));
    const long long xc = (VOF_S(-1, 0, -1) + VOF_S(0, 0, -1) + VOF_S(1, 0, -1)) -
                         (VOF_S(-1, 0, 1) + VOF_S(0, 0, 1) + VOF_S(1, 0, 1));
    const long long yb = (VOF_S(-1, -1, 0) + VOF_S(-1, 0, 0) + VOF_S(-1, 1, 0)) -
                         (VOF_S(1, -1, 0) + VOF_S(1, 0, 0) + VOF_S(1, 1, 0));
    const long long yc = (VOF_S(0, -1, -1) + VOF_S(0, 0, -1) + VOF_S(0, 1, -1)) -
                         (VOF_S(0, -1, 1) + VOF_S(0, 0, 1) + VOF_S(0, 1, 1));
    const long long zb = (VOF_S(-1, 0, -1) + VOF_S(-1, 0, 0) + VOF_S(-1, 0, 1)) -
                         (VOF_S(1, 0, -1) + VOF_S(1, 0, 0) + VOF_S(1, 0, 1));
    const long long zc = (VOF_S(0, -1, -1) + VOF_S(0, -1, 0) + VOF_S(0, -1, 1)) -
                         (VOF_S(0, 1, -1) + VOF_S(0, 1, 0) + VOF_S(0, 1, 1));
#undef VOF_S
    // T of each candidate, compared in units of 2^-52; near a tie by the
    // rounded quotients of the rule (ties to the lower axis)
    const int sh = eref - 1081;  // half of one unit is 2^sh
    const int k52 = 1028 - eref, kq = k52 > 63 ? 63 : (k52 < 0 ? 0 : k52);
    const unsigned long long tx = mag64(xb) + mag64(xc), ty = mag64(yb) + mag64(yc), tz = mag64(zb) + mag64(zc);
    auto l1_of = [&](int axis) {  // the norm with every sum rounded in the rule's order
        const int sa = axis == 0 ? 1 : (axis == 1 ? 3 : 9), sb = axis == 0 ? 3 : 1, sc = axis == 2 ? 3 : 9;
        auto column = [&](int o) { return (st[13 + o - sa] + st[13 + o]) + st[13 + o + sa]; };
        const double b = abs64((column(-sb) - column(sb)) * 0.5), c = abs64((column(-sc) - column(sc)) * 0.5);
        return axis == 0 ? (1.0 + b) + c : (axis == 1 ? (b + 1.0) + c : (b + c) + 1.0);
    };
    auto better = [&](unsigned long long t_new, int a_new, unsigned long long t_best, int a_best) {
        const long long d = (long long)(t_best >> kq) - (long long)(t_new >> kq);
        if (d > 4) return true;
        if (d < -4) return false;
        const double l_new = l1_of(a_new), l_best = l1_of(a_best);
        const long long u = bits64(l_best) - bits64(l_new);  // (a quotient falls as its norm rises)
        return u > 2 || (u > 0 && 1.0 / l_new > 1.0 / l_best);
    };
    int axis = 0;
    unsigned long long t = tx;
    if (better(ty, 1, t, axis)) { axis = 1; t = ty; }
    if (better(tz, 2, t, axis)) { axis = 2; t = tz; }
    // Youngs where ymax / ny < 1 / (1 + T/2): ymax T/2 < ny - ymax
    const unsigned long long ax = mag64(y[0]), ay = mag64(y[1]), az = mag64(y[2]);
    unsigned long long ymax = ax > ay ? ax : ay;
    ymax = ymax > az ? ymax : az;
    const unsigned long long rest = ax + ay + az - ymax;
    bool youngs = false;
    // (the rule's ny >= 1e-30: one unit, 2^(eref - 1080), reaches it from eref = 981)
    const double ny = (double)(ax + ay + az);  // below 2^63.6
    if (ymax != 0 && (eref >= 981 || le_pos(1e-30, from_bits64(bits64(ny) + ((long long)(eref - 1080) << 52))))) {
#ifdef __CUDA_ARCH__
        const float half_t = __ull2float_rn(t) * __int_as_float((sh + 127 < 1 ? 0 : sh + 127) << 23);
        const float lf = __ull2float_rn(ymax) * half_t, rf = __ull2float_rn(rest);
#else
        const float half_t = sh + 127 < 1 ? 0.f : ldexpf((float)t, sh);
        const float lf = (float)ymax * half_t, rf = (float)rest;
#endif
        youngs = lf < rf;
        if (fabsf(lf - rf) <= 1e-5f * (lf + rf)) youngs = (double)ymax * scaled64((long long)t, sh) < (double)rest;
    }
    if (youngs) {  // the largest component to 1 .. 2
#ifdef __CUDA_ARCH__
        const int top = __clzll((long long)ymax) - 63;
#else
        const int top = __builtin_clzll(ymax) - 63;
#endif
        m[0] = scaled64(y[0], top);
        m[1] = scaled64(y[1], top);
        m[2] = scaled64(y[2], top);
        return;
    }
    const long long db = axis == 0 ? xb : (axis == 1 ? yb : zb), dc = axis == 0 ? xc : (axis == 1 ? yc : zc);
    const double own = (axis == 0 ? y[0] : (axis == 1 ? y[1] : y[2])) < 0 ? -1.0 : 1.0;
    const double mb = scaled64(db, sh), mc = scaled64(dc, sh);
    m[0] = axis == 0 ? own : mb;
    m[1] = axis == 1 ? own : (axis == 0 ? mb : mc);
    m[2] = axis == 2 ? own : mc;
}

// The swept slab of a face flux mapped onto the unit cube.  In the frame
// reflected to non-negative components n the slab [1 - s, 1] (s > 0) or
// [0, |s|] (s < 0) keeps or swaps its end with the sign of m_d; then n_d ->
// n_d |s|, alpha -> alpha - n_d x0.  n: sorted on return; returns the constant.
VOF_HD double slab64(const double m[3], double al, int d, double s, double n[3]) {
    n[0] = abs64(m[0]);
    n[1] = abs64(m[1]);
    n[2] = abs64(m[2]);
    const double as = abs64(s);
    const double nd = d == 0 ? n[0] : (d == 1 ? n[1] : n[2]), md = d == 0 ? m[0] : (d == 1 ? m[1] : m[2]);
    const bool far_end = negative64(s) == negative64(md);
    const double x = far_end ? fma(-nd, 1.0 - as, al) : al;
    const double sd = nd * as;
    if (d == 0) n[0] = sd;
    else if (d == 1) n[1] = sd;
    else n[2] = sd;
    sort3_pos(n[0], n[1], n[2]);
    return x;
}

// Flux through a face of the donor of fraction cv in (0, 1) with normal
// direction m (largest component within 2^-20 .. 2^20); s is the signed
// Courant number.
VOF_HD double face_flux64(const double m[3], double cv, int d, double s) {
    double a = abs64(m[0]), b = abs64(m[1]), c = abs64(m[2]);
    sort3_pos(a, b, c);
    double n[3];
    const double x = slab64(m, alpha64(a, b, c, cv), d, s, n);
    if (!lt_pos(0.0, n[2])) return bits64(x) > 0 ? s : 0.0;
    return s * vol64(n[0], n[1], n[2], x);
}

}  // namespace vof
