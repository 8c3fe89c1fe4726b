"""The FP64 plane constant and face flux (csrc/plic64.cuh), compiled for the host,
against 113-bit arithmetic: random planes (components down to 1e-6 of the largest,
or zero), fractions down to 1e-12 from 0 and 1, Courant numbers of both signs.

The references take the volume by inclusion-exclusion over the vertices, whose
cancellation costs 113-bit numbers at most 1e-34 / (1e-6)^2; the constant by
bisection and Newton on it.  Bounds, with |m|_1 = 1: a constant is a root of a
formula of some ten operations on numbers up to 1, each rounded by 2^-53, and a
flux, of |s| <= 1/2, a volume that the constant's error reaches with a slope of at
most 3 / 2 per unit: 10 * 2^-53 for both, 1.2e-15.  The errors found are printed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_07463_gb300", "csrc")
SOURCE = r"""
#include "plic64.cuh"
#if __LDBL_MANT_DIG__ >= 113
typedef long double quad;
#else
typedef __float128 quad;
#endif
using namespace vof;

// volume of {x in the unit cube: m.x < al}, m >= 0
static quad volume(const quad* m, quad al) {
    quad c[3], S = 0, p = 1, v = 0;
    int n = 0;
    for (int a = 0; a < 3; ++a)
        if (m[a] > 0) c[n++] = m[a], S += m[a], p *= m[a] * n;
    if (al <= 0) return 0;
    if (al >= S) return 1;
    const bool flip = al > S - al;
    if (flip) al = S - al;
    for (int b = 0; b < 1 << n; ++b) {
        quad t = al;
        int sign = 1;
        for (int a = 0; a < n; ++a)
            if (b >> a & 1) t -= c[a], sign = -sign;
        if (t <= 0) continue;
        quad q = sign;
        for (int a = 0; a < n; ++a) q *= t;
        v += q;
    }
    v /= p;
    return flip ? 1 - v : v;
}
static quad constant(const quad* m, quad c) {
    quad lo = 0, hi = m[0] + m[1] + m[2];
    for (int i = 0; i < 125; ++i) {
        const quad mid = (lo + hi) / 2;
        (volume(m, mid) < c ? lo : hi) = mid;
    }
    return hi;
}
static quad magnitude(quad v) { return v < 0 ? -v : v; }

// err[0], err[1]: error of the constant (m >= 0, |m|_1 = 1) and of the flux
extern "C" void errors(const double* mm, const double* cc, const double* ss, int n, double* err) {
    for (int i = 0; i < n; ++i) {
        const double *m = mm + 3 * i, c = cc[i], s = ss[i];
        const int d = i % 3;
        double a = abs64(m[0]), b = abs64(m[1]), e = abs64(m[2]);
        sort3_pos(a, b, e);
        const bool flip = lt_pos(0.5, c);
        const double x = alpha64_half(a, b, e, flip ? 1.0 - c : c), al = flip ? (a + b + e) - x : x;
        const double f = face_flux64_at(m, al, d, s);
        quad q[3];
        for (int k = 0; k < 3; ++k) q[k] = abs64(m[k]);
        const quad want = constant(q, c), as = s < 0 ? -(quad)s : (quad)s;
        err[2 * i] = (double)magnitude((quad)al - want);
        // the swept end of the cube in the frame of non-negative components
        const bool far_end = (s > 0) == (m[d] >= 0);
        const quad cut = far_end ? want - q[d] * (1 - as) : want;
        q[d] *= as;
        err[2 * i + 1] = (double)magnitude((quad)f - (quad)s * volume(q, cut));
    }
}
"""


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    d = tmp_path_factory.mktemp("plic64")
    (d / "host.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-x", "c++",
                    str(d / "host.cpp"), "-o", str(d / "host.so")], check=True)
    fn = ctypes.CDLL(str(d / "host.so")).errors
    ptr = np.ctypeslib.ndpointer(np.float64, flags="C_CONTIGUOUS")
    fn.argtypes, fn.restype = [ptr, ptr, ptr, ctypes.c_int, ptr], None

    def run(m, c, s):
        out = np.empty((len(c), 2))
        fn(np.ascontiguousarray(m), c, s, len(c), out)
        return out

    return run


def test_errors(errors):
    n = int(os.environ.get("VOF_QUAD_PLANES", "20000"))
    rng = np.random.default_rng(1)
    m = rng.normal(size=(n, 3))
    m *= 10.0 ** (rng.uniform(-6, 0, (n, 3)) * (rng.random((n, 3)) < 0.3))
    m[rng.random((n, 3)) < 0.03] = 0.0
    m[~m.any(1)] = 1.0
    m /= np.abs(m).sum(1, keepdims=True)
    m[np.abs(m) < 1e-6 * np.abs(m).max(1, keepdims=True)] = 0.0
    c = rng.random(n)
    edge = rng.random(n) < 0.2
    c[edge] = 10.0 ** rng.uniform(-12, 0, int(edge.sum()))
    top = rng.random(n) < 0.1
    c[top] = 1.0 - 10.0 ** rng.uniform(-12, -1, int(top.sum()))
    c = np.clip(c, 1e-12, 1.0 - 1e-12)
    s = rng.uniform(-0.5, 0.5, n)
    err = errors(m, c, s)
    print("\nconstant: max %.2e mean %.2e; flux: max %.2e mean %.2e" % (err[:, 0].max(), err[:, 0].mean(),
                                                                      err[:, 1].max(), err[:, 1].mean()))
    assert err.max() <= 10 * 2.0 ** -53
