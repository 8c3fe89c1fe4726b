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
// Against 113-bit arithmetic on a million random planes, fractions and Courant
// numbers (tests/test_plic64_quad.py with a million planes; it takes 20000):
// flux within 3.9e-16 (mean 1.08e-17), plane constant within 3.0e-16 (mean
// 3.1e-17); the piecewise Gauss evaluation and its Newton inversion that stood
// here before gave 3.9e-16 (1.31e-17) and 3.7e-16 (4.1e-17) on the same planes.
// Times: k_face_flux_bx.
#pragma once

#include <math.h>
#include <stdint.h>

#include "myc.cuh"

namespace vof {

#ifdef __CUDACC__
#define VOF_HD_CALL static __host__ __device__ __noinline__
#else
#define VOF_HD_CALL static
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

// Conversions on the integer ALU (the FP64 unit does them otherwise).  The
// float of v >= 0, cut off instead of rounded: 0 below FP32's normal range, v
// below 2^127.
VOF_HD float low_float(double v) {
    const long long b = bits64(v) - (896LL << 52);
    const int f = b < (1LL << 52) ? 0 : (int)(b >> 29);
#ifdef __CUDA_ARCH__
    return __int_as_float(f);
#else
    float r;
    __builtin_memcpy(&r, &f, 4);
    return r;
#endif
}
// The double of a float that is positive and normal.
VOF_HD double wide(float v) {
#ifdef __CUDA_ARCH__
    const int f = __float_as_int(v);
#else
    int f;
    __builtin_memcpy(&f, &v, 4);
#endif
    return from_bits64(((long long)f << 29) + (896LL << 52));
}

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
    const float yf = cbrtf(low_float(m));
    const double r = wide(1.f / (3.f * yf * yf));
    double y = wide(yf);
    y = fma(-fma(y * y, y, -m), r, y);
    y = fma(-fma(y * y, y, -m), r, y);
    return y * from_bits64((long long)(1023 + k) << 52);
}

// Volume under the plane a x + b y + c z < x in the unit cube, sorted
// 0 <= a <= b <= c, c > 0, 0 <= x <= (a + b + c) / 2: numerator and divisor of
// every piece, taken by selects (19 products and sums; as branches the lanes of
// a warp paid for 24 and the branches).
VOF_HD double vol64_half(double a, double b, double c, double x) {
    const double ab = a + b, e = 6.0 * b * c, ea = e * a;
    const double tb = x - b, tc = plus64(x - c);
    const double q = fma(3.0 * x, x - a, a * a);
    const bool tip = le_pos(x, a);
    const bool prism = lt_pos(ab, x);          // (x <= S/2 leaves it to c > a + b)
    const bool corner = lt_pos(b, x);          // not at x = b, where a may be zero
    double num = corner ? fma(a, q, -fma(tb * tb, tb, tc * tc * tc)) : q;
    double den = corner ? ea : e;
    num = prism ? fma(2.0, x, -ab) : num;
    den = prism ? 2.0 * c : den;
    num = tip ? x * x * x : num;
    den = tip ? ea : den;
    // a divisor this small belongs to a plane whose volume is below 1e-90
    return lt_pos(den, 1e-290) ? 0.0 : num / den;
}

// The same for any x; S = a + b + c > 0.
VOF_HD double vol64(double a, double b, double c, double x) {
    if (bits64(x) <= 0) return 0.0;
    const double S = a + b + c, y = S - x;
    if (bits64(y) <= 0) return 1.0;
    const bool flip = lt_pos(y, x);  // (one copy of the pieces for both halves)
    const double v = vol64_half(a, b, c, flip ? y : x);
    return flip ? 1.0 - v : v;
}

// Root x in (0, S/2] of vol64_half(a, b, c, x) = v, 0 < v <= 1/2, sorted
// 0 <= a <= b <= c, c > 0.  In units of b (p = a/b, w = c v / b, g = c/b):
//   6w <= p^2:            x^3 = 6 p w
//   6w <= 3 - 3p + p^2:   3x(x - p) + p^2 = 6w
//   c >= a + b, 2w >= 1 + p:  the prism, x = w + (1 + p)/2
//   else  p (3x(x - p) + p^2 - 6w) = (x - 1)^3 + (x - g)_+^3, seeded by the
//   middle root of the cubic in trigonometric form (alpha_sorted_pw).
enum AlphaPiece { kAlphaCubic = 0, kAlphaSqrt = 1, kAlphaCbrt = 2, kAlphaLinear = 3 };
// 1 / b for b within FP32's range: two Newton steps from the FP32 quotient.
VOF_HD double rcp64(double b) {
    double r = wide(1.f / low_float(b));
    r = fma(fma(-b, r, 1.0), r, r);
    return fma(fma(-b, r, 1.0), r, r);
}
// The piece the root lies in with its variables p, w6 = 6w and g; root / b is
// alpha64_root of these, the linear pieces' root is x.  c within 2^-20 .. 2^20.
VOF_HD int alpha64_piece(double a, double b, double c, double v, double& p, double& w6, double& g, double& x) {
    const double cv = c * v;
    x = cv;
    p = w6 = g = 0.0;
    if (lt_pos(b, 1e-30 * c)) return kAlphaLinear;  // a plane across one axis (off by < 1e-30 c)
    const double ib = rcp64(b);
    p = a * ib;
    w6 = 6.0 * cv * ib;
    g = c * ib;
    const double p2 = p * p;
    if (le_pos(w6, p2)) return kAlphaCbrt;
    if (!negative64(fma(3.0, 1.0 - p, p2) - w6)) return kAlphaSqrt;
    const double ab = a + b;
    if (le_pos(ab, c) && le_pos(ab, 2.0 * cv)) {
        x = fma(0.5, ab, cv);
        return kAlphaLinear;
    }
    return kAlphaCubic;
}
VOF_HD double alpha64_cubic(double p, double w6, double g) {
    // seed
    const float pf = low_float(p), gf = low_float(g), wf = low_float(w6) * (1.f / 6.f);
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
    double x = xf > 1.f ? wide(xf) : 1.0;  // (1 also for a NaN of a degenerate seed)
    if (lt_pos(hi, x)) x = hi;
    if (lt_pos(p, 1e-20)) return x;  // the region is narrower than an ulp
    // Newton: G(x) = p (3x(x - p) + p^2 - 6w) - (x - 1)^3 - (x - g)_+^3
    const float xs = low_float(x), t1 = xs - 1.f, t2 = fmaxf(xs - gf, 0.f);
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
    return lt_pos(hi, x) ? hi : x;
}
VOF_HD double alpha64_root(int piece, double p, double w6, double g) {
    if (piece == kAlphaCubic) return alpha64_cubic(p, w6, g);
    if (piece == kAlphaSqrt) return 0.5 * (p + sqrt(fma(-1.0 / 3.0, p * p, (4.0 / 3.0) * w6)));
    return cbrt64(p * w6);
}
VOF_HD double alpha64_half(double a, double b, double c, double v) {
    double p, w6, g, x;
    const int piece = alpha64_piece(a, b, c, v, p, w6, g, x);
    return piece == kAlphaLinear ? x : b * alpha64_root(piece, p, w6, g);
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
VOF_HD unsigned long long mag64(long long v) { return (unsigned long long)(v < 0 ? -v : v); }
VOF_HD int clz64(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}
// A whole number times 2^sh as a double, rounded to 53 bits (0 stays 0).
VOF_HD double scaled64(long long n, int sh) {
    const unsigned long long u = mag64(n);
    if (u == 0) return 0.0;
    const int lz = clz64(u);
    const unsigned long long top = u << lz;
    const long long r = (long long)((top >> 11) + ((top >> 10) & 1));  // 2^52 .. 2^53
    const long long b = r + ((long long)(1085 - lz + sh) << 52);
    return from_bits64(n < 0 ? b | (long long)0x8000000000000000ULL : b);
}

// The rule evaluated in double, for the stencils below: as it stands, and for
// values of fractions' size (a few divisions instead of seven: quotients are
// formed only where rounding may decide, and a common factor is left in).
VOF_HD_CALL void myc_rule64(const double* st, double m[3]) { myc_normal<double>(st, m); }
VOF_HD_CALL void myc_tie64(const double* st, double m[3]) {
    double y[3];
    youngs_raw(st, y);
    centred_column(st, 0, y, m);
    double l = l1norm(m);
VOF_UNROLL
    for (int a = 1; a < 3; ++a) {
        double r[3];
        centred_column(st, a, y, r);
        const double n = l1norm(r);
        // 1 / n > 1 / l, which differ if n and l do by two ulps
        if (n < l && (l - n > 5e-16 * l || 1.0 / n > 1.0 / l)) {
            l = n;
            m[0] = r[0];
            m[1] = r[1];
            m[2] = r[2];
        }
    }
    const double ny = l1norm(y);
    if (!(ny >= 1e-30)) return;
    const double y01 = lt_pos(abs64(y[0]), abs64(y[1])) ? abs64(y[1]) : abs64(y[0]);
    const double ymax = lt_pos(y01, abs64(y[2])) ? abs64(y[2]) : y01;
    const double gap = ny - ymax * l;  // ymax / ny < 1 / l
    if (abs64(gap) > 1e-14 * ny ? gap > 0.0 : ymax / ny < 1.0 / l) {
        const double il = 1.0 / ny;
        m[0] = y[0] * il;
        m[1] = y[1] * il;
        m[2] = y[2] * il;
    }
}

// Mixed-Youngs-Centred direction of a stencil (myc.cuh gives the rule), not
// normalised: its largest component lies in 1/3 .. 96.  The hundred additions run
// on 64-bit integers (the integer pipes are idle in the FP64 kernels): the
// fractions become whole numbers of 2^-57 of the largest neighbour's binade, 32
// times finer than that value's own last place, so that sums and differences are
// exact and no less accurate than in double.  The candidates compare by T, their
// L1 norm being 1 + T/2, Youngs against the best candidate in float.
//
// The rule in double rounds its sums, so that near a tie it may decide otherwise
// than exact sums do, and what it decides there moves a normal by any angle.
// Where a decision (which candidate, Youngs or not, the sign of the own
// component) lies within a bound on that rounding, where the values are too far
// from fractions for the common unit, and beside an infinity or a NaN, the rule
// itself is evaluated.  The bounds: Youngs' sums of 18 terms, 64 of the largest
// value in all, round by less than 18 x 64 x 2^-53 of it, 2^15 units, a column
// candidate's norm by less than 16 x 2^-52.
//
// edge: an open decision is left to the exact sums where the centre lies within
// it of 0 or 1.  A flux changes by no more than that; inside a drop, where a sweep
// leaves fractions a few ulps below 1, one interfacial cell in eight has an open
// decision, elsewhere one in ten thousand (a step of the 256^3, K = 8, phi = 0.3
// box takes 4.7 ms, and 6.7 ms with the rule for all of them).
constexpr double kFluxEdge = 3.5527136788005009e-15;  // 2^-48
VOF_HD void myc_direction64(const double* st, double m[3], double edge) {
#define VOF_S(i, j, k) q[((k) + 1) * 9 + ((j) + 1) * 3 + ((i) + 1)]
    int eref = 600;  // (the unit of values below 2^-423)
    long long any = 0;  // the neighbours' bits
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 27; ++c) {
        const int e = (int)(bits64(st[c]) >> 52) & 0x7ff;
        if (c != 13) {  // (the centre enters no sum)
            eref = e > eref ? e : eref;
            any |= bits64(st[c]) << 1;
        }
    }
    if (eref >= 1028) {  // values of 32 and more, an infinity or a NaN
        myc_rule64(st, m);
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
    // T of each candidate (ties to the lower axis).  Below 2^-54 every norm
    // rounds to 1: the lowest axis.
    const int sh = eref - 1081;  // half of one unit is 2^sh
    const unsigned long long tx = mag64(xb) + mag64(xc), ty = mag64(yb) + mag64(yc), tz = mag64(zb) + mag64(zc);
    const bool flat = (tx | ty | tz) >> (eref > 1026 ? 0 : (eref < 964 ? 62 : 1026 - eref)) == 0;
    const int axis = flat || (tx <= ty && tx <= tz) ? 0 : (ty <= tz ? 1 : 2);
    const unsigned long long t = axis == 0 ? tx : (axis == 1 ? ty : tz);
    const unsigned long long t1 = axis == 0 ? ty : tx, t2 = axis == 2 ? ty : tz;
    // (32 x 2^-52 in units; 64 bits hold every T)
    const unsigned long long slack = 1ull << (eref > 1033 ? 0 : (eref < 970 ? 63 : 1033 - eref));
    bool open = !flat && ((t1 < t2 ? t1 : t2) - t <= slack);
    // Youngs where ymax / ny < 1 / (1 + T/2): ymax T/2 < ny - ymax
    const unsigned long long ax = mag64(y[0]), ay = mag64(y[1]), az = mag64(y[2]);
    unsigned long long ymax = ax > ay ? ax : ay;
    ymax = ymax > az ? ymax : az;
    const unsigned long long rest = ax + ay + az - ymax;
    bool youngs = false;
    // (the rule's |y|_1 >= 1e-30: one unit, 2^(eref - 1080), reaches it from eref = 981)
    if (ymax != 0 && (eref >= 981 || le_pos(1e-30, scaled64((long long)((ymax + rest) >> 2), eref - 1078)))) {
#ifdef __CUDA_ARCH__
        const float half_t = __ull2float_rn(t) * __int_as_float((sh + 127 < 1 ? 0 : sh + 127) << 23);
        const float lf = __ull2float_rn(ymax) * half_t, rf = __ull2float_rn(rest);
#else
        const float half_t = sh + 127 < 1 ? 0.f : ldexpf((float)t, sh);
        const float lf = (float)ymax * half_t, rf = (float)rest;
#endif
        youngs = lf < rf;
        open = open || fabsf(lf - rf) <= 1e-5f * (lf + rf) + 131072.f;
    }
    // (Youngs' rounding within 2^-21 of its largest component)
    const unsigned long long own_y = axis == 0 ? ax : (axis == 1 ? ay : az);
    open = open || ymax < (1ull << 36) || (!youngs && own_y < (1ull << 15));
    if (open && any != 0 && le_pos(edge, plus64(st[13])) && le_pos(edge, plus64(1.0 - st[13]))) {
        myc_tie64(st, m);
        return;
    }
    // Youngs' largest component goes to 1 .. 2
    const long long cb = axis == 0 ? xb : (axis == 1 ? yb : zb), cc = axis == 0 ? xc : (axis == 1 ? yc : zc);
    const int ms = youngs ? clz64(ymax) - 63 : sh;
    const double m0 = scaled64(youngs ? y[0] : cb, ms), m1 = scaled64(youngs ? y[1] : cc, ms);
    if (youngs) {
        m[0] = m0;
        m[1] = m1;
        m[2] = scaled64(y[2], ms);
        return;
    }
    const double own = (axis == 0 ? y[0] : (axis == 1 ? y[1] : y[2])) < 0 ? -1.0 : 1.0;
    m[0] = axis == 0 ? own : m0;
    m[1] = axis == 1 ? own : (axis == 0 ? m0 : m1);
    m[2] = axis == 2 ? own : m1;
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

// Flux through a face of the donor cut by the plane of direction m (largest
// component within 2^-20 .. 2^20) and constant al in the reflected frame; s is
// the signed Courant number.
VOF_HD double face_flux64_at(const double m[3], double al, int d, double s) {
    double n[3];
    const double x = slab64(m, al, d, s, n);
    if (!lt_pos(0.0, n[2])) return bits64(x) > 0 ? s : 0.0;
    return s * vol64(n[0], n[1], n[2], x);
}

}  // namespace vof
