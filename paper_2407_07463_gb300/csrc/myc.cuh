// The Mixed-Youngs-Centred rule (Section 2.2): FP32 normals, and the double
// normals of stencils whose decisions the integer sums of plic64.cuh leave open.
#pragma once

#include <math.h>

namespace vof {

#ifdef __CUDACC__
#define VOF_HD __host__ __device__ __forceinline__
#define VOF_UNROLL _Pragma("unroll")
#else
#define VOF_HD static inline
#define VOF_UNROLL
#endif

// Normals.  Stencil st[(k+1)*9 + (j+1)*3 + (i+1)], offsets i (x), j (y), k (z).

#define VOF_ST(st, i, j, k) ((st)[((k) + 1) * 9 + ((j) + 1) * 3 + ((i) + 1)])

template <typename T>
VOF_HD void youngs_raw(const T* st, T y[3]) {
    const T W[3] = {T(1), T(2), T(1)};
    T yx = T(0), yy = T(0), yz = T(0);
VOF_UNROLL
    for (int b = -1; b <= 1; ++b)
VOF_UNROLL
        for (int a = -1; a <= 1; ++a) {
            T w = W[a + 1] * W[b + 1];
            yx += w * (VOF_ST(st, -1, a, b) - VOF_ST(st, 1, a, b));
            yy += w * (VOF_ST(st, a, -1, b) - VOF_ST(st, a, 1, b));
            yz += w * (VOF_ST(st, a, b, -1) - VOF_ST(st, a, b, 1));
        }
    y[0] = yx;
    y[1] = yy;
    y[2] = yz;
}

template <typename T>
VOF_HD T l1norm(const T v[3]) {
    return fabs(v[0]) + fabs(v[1]) + fabs(v[2]);
}

template <typename T>
VOF_HD T st_axis(const T* st, int axis, int t, int p, int q) {
    // p along the lower of the two other axes, q along the higher
    if (axis == 0) return VOF_ST(st, t, p, q);
    if (axis == 1) return VOF_ST(st, p, t, q);
    return VOF_ST(st, p, q, t);
}

// Centred-column candidate along `axis` (not normalised).
template <typename T>
VOF_HD void centred_column(const T* st, int axis, const T y[3], T m[3]) {
    T H[3][3];
VOF_UNROLL
    for (int p = -1; p <= 1; ++p)
VOF_UNROLL
        for (int q = -1; q <= 1; ++q)
            H[p + 1][q + 1] = st_axis(st, axis, -1, p, q) + st_axis(st, axis, 0, p, q) +
                              st_axis(st, axis, 1, p, q);
    int b = axis == 0 ? 1 : 0;
    int c = axis == 2 ? 1 : 2;
    m[b] = (H[0][1] - H[2][1]) * T(0.5);
    m[c] = (H[1][0] - H[1][2]) * T(0.5);
    m[axis] = y[axis] < T(0) ? T(-1) : T(1);
}

// Mixed-Youngs-Centred normal (L1-normalised, pointing out of the c = 1
// phase).  Among the three centred-column candidates the one with the
// largest own-axis component |m_a|/|m|_1 is kept (ties to the lower axis);
// the Youngs normal (average of the eight vertex gradients) replaces it when
// its largest |component|/|m|_1 is strictly smaller -- saturated columns make
// a centred-column normal look more grid-aligned than it is.
template <typename T>
VOF_HD void myc_normal(const T* st, T m[3]) {
    T y[3];
    youngs_raw(st, y);
    T best[3] = {T(0), T(0), T(0)};
    T best_own = T(-1);
VOF_UNROLL
    for (int a = 0; a < 3; ++a) {
        T r[3];
        centred_column(st, a, y, r);
        T own = fabs(r[a]) / l1norm(r);
        if (own > best_own) {
            best_own = own;
            best[0] = r[0];
            best[1] = r[1];
            best[2] = r[2];
        }
    }
    T ny = l1norm(y);
    if (ny >= T(1e-30)) {
        T ymax = fabs(y[0]);
        if (fabs(y[1]) > ymax) ymax = fabs(y[1]);
        if (fabs(y[2]) > ymax) ymax = fabs(y[2]);
        if (ymax / ny < best_own) {
            m[0] = y[0] / ny;
            m[1] = y[1] / ny;
            m[2] = y[2] / ny;
            return;
        }
    }
    T n = l1norm(best);
    m[0] = best[0] / n;
    m[1] = best[1] / n;
    m[2] = best[2] / n;
}

}  // namespace vof
