// Curvature of each colour field by height functions and the surface-tension
// source f = sum_i gamma kappa_i grad C_i (Section 2.3: with N(t) tracers
// the capillary force is the sum of every tracer's contribution, each with
// its own curvature computed as for a single tracer).
//
// Curvature of an interfacial cell (0 < c < 1): the axis a of the largest
// |component| of the cell's Mixed-Youngs-Centred normal (ties to the lower
// axis); the 3x3 columns of 7 cells along a (offsets -3..3) centred on the
// cell and its neighbours across a hold the heights H = sum of c.  Every
// column must contain the interface -- its end on the c = 1 side (opposite
// the normal) above 1/2, the other end below 1/2 -- else the cell has no
// curvature (NaN).  With f_x, f_y, f_xx, f_yy, f_xy the centred
// differences of H (cell units),
//   kappa = -[f_xx (1 + f_y^2) + f_yy (1 + f_x^2) - 2 f_xy f_x f_y]
//           / (1 + f_x^2 + f_y^2)^(3/2) / h,
// the divergence of the normal pointing out of the c = 1 phase (2/R for a
// drop of radius R).
//
// Interfacial cells are few (2% of a field at phi = 0.25 in 7 fields) and
// cost 90 gathers each: a block scans a tile of consecutive cells with 16-byte
// loads, collects the interfacial ones in shared memory and then takes them a
// thread each, on full warps.  Measured, 192^3 and 7 fields in FP32: 0.11 ms
// for the curvatures and 0.16 ms for the source (0.18 ms with three fields'
// values held in flight: fewer warps); a thread per cell took 2.19 ms for the
// curvatures (few lanes of a warp gathering, an index modulo per value) and
// 0.40 ms for the source.  In double 0.48 and 1.12 ms, bound by FP64 issue.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "plic.cuh"
#include "update_vec.cuh"

namespace vof {

template <typename T>
__device__ __forceinline__ T nan_of();
template <>
__device__ __forceinline__ double nan_of<double>() { return __longlong_as_double(0x7ff8000000000000LL); }
template <>
__device__ __forceinline__ float nan_of<float>() { return __int_as_float(0x7fc00000); }

// Offset of the cell t away from p on an axis of n cells (periodic; any t).
__device__ __forceinline__ int axis_step(int p, int t, int n) {
    int q = p + t;
    if (q >= n || q < 0) q = wrapi(q, n);
    return q - p;
}

template <typename T>
__device__ __forceinline__ T cell_curvature(const T* __restrict__ cf, const Dims& g, int x, int i, int j, int k, T h) {
    const int sx = 1, sy = g.nx, sz = g.nx * g.ny;
    T st[27];
    {
        const int ox[3] = {axis_step(i, -1, g.nx) * sx, 0, axis_step(i, 1, g.nx) * sx};
        const int oy[3] = {axis_step(j, -1, g.ny) * sy, 0, axis_step(j, 1, g.ny) * sy};
        const int oz[3] = {axis_step(k, -1, g.nz) * sz, 0, axis_step(k, 1, g.nz) * sz};
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int a = 0; a < 3; ++a) st[c * 9 + b * 3 + a] = cf[x + ox[a] + oy[b] + oz[c]];
    }
    T m[3];
    myc_normal(st, m);
    int a = 0;
    T ma = m[0];
    if (fabs(m[1]) > fabs(ma)) { a = 1; ma = m[1]; }
    if (fabs(m[2]) > fabs(ma)) { a = 2; ma = m[2]; }
    const bool up = ma < T(0);  // the c = 1 side lies at +3
    // steps along the height axis a and across it (b < e)
    const int pa = a == 0 ? i : (a == 1 ? j : k), na = a == 0 ? g.nx : (a == 1 ? g.ny : g.nz);
    const int sa = a == 0 ? sx : (a == 1 ? sy : sz);
    const int pb = a == 0 ? j : i, nb = a == 0 ? g.ny : g.nx, sb = a == 0 ? sy : sx;
    const int pe = a == 2 ? j : k, ne = a == 2 ? g.ny : g.nz, se = a == 2 ? sy : sz;
    int oa[7];
#pragma unroll
    for (int t = -3; t <= 3; ++t) oa[t + 3] = axis_step(pa, t, na) * sa;
    const int ob[3] = {axis_step(pb, -1, nb) * sb, 0, axis_step(pb, 1, nb) * sb};
    const int oe[3] = {axis_step(pe, -1, ne) * se, 0, axis_step(pe, 1, ne) * se};
    T H[3][3];
    bool ok = true;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const T* col = cf + x + ob[p] + oe[q];
            const T first = col[oa[0]], last = col[oa[6]];
            T sum = first;
#pragma unroll
            for (int t = 1; t < 6; ++t) sum += col[oa[t]];
            H[p][q] = sum + last;
            ok = ok && (up ? last : first) > T(0.5) && (up ? first : last) < T(0.5);
        }
    if (!ok) return nan_of<T>();
    const T fx = T(0.5) * (H[2][1] - H[0][1]), fy = T(0.5) * (H[1][2] - H[1][0]);
    const T fxx = H[2][1] - T(2) * H[1][1] + H[0][1], fyy = H[1][2] - T(2) * H[1][1] + H[1][0];
    const T fxy = T(0.25) * (H[2][2] - H[2][0] - H[0][2] + H[0][0]);
    const T g2 = T(1) + fx * fx + fy * fy;
    return -(fxx * (T(1) + fy * fy) + fyy * (T(1) + fx * fx) - T(2) * fxy * fx * fy) / (g2 * sqrt_t(g2)) / h;
}

template <typename T>
__device__ __forceinline__ bool interfacial(T v) { return v > T(0) && v < T(1); }
template <>
__device__ __forceinline__ bool interfacial(double v) {  // the open interval on the bit pattern (no FP64 issue)
    const long long b = __double_as_longlong(v);
    return b > 0 && b < 0x3FF0000000000000LL;
}

// Whether a value other than 0 and 1 is among those seen: between two such cells
// nothing is added, whatever their neighbours are.  (In double by words: the low
// ones join in one word, two to an instruction.)
struct Unsettled32 {
    bool any;
    __device__ __forceinline__ void see(float v) { any = any || !(v == 0.f || v == 1.f); }
    __device__ __forceinline__ bool found() const { return any; }
};
struct Unsettled64 {
    bool any;
    int low = 0;
    __device__ __forceinline__ void see(double v) {
        const int hi = __double2hiint(v);
        low |= __double2loint(v);
        any = any || !(hi == 0 || hi == 0x3FF00000);
    }
    __device__ __forceinline__ bool found() const { return any || low != 0; }
};
// v is finite (in double without an FP64 compare).
__device__ __forceinline__ bool finite_bits(float v) { return isfinite(v); }
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000; }
// acc + zero * (p - q), zero being 0 (or a NaN): changes acc only where the
// difference is not finite.  In double a difference below 2^1023 is.
__device__ __forceinline__ void add_nothing(float& acc, float zero, bool, float p, float q) { acc += zero * (p - q); }
__device__ __forceinline__ void add_nothing(double& acc, double zero, bool all, double p, double q) {
    if (all || max(__double2hiint(p) & 0x7FFFFFFF, __double2hiint(q) & 0x7FFFFFFF) >= 0x7FD00000) acc += zero * (p - q);
}

// Curvatures of the fields blockIdx.y of c ([K][N]) into kappa: NaN in every
// cell without one if FILL, else only the interfacial cells are written.
constexpr int kCurvThreads = 256;

template <typename T, int VW, bool FILL, int TILE>
__global__ void __launch_bounds__(kCurvThreads) k_curvature(const T* __restrict__ c, Dims g, T h,
                                                            T* __restrict__ kappa) {
    __shared__ uint16_t s_cell[TILE];
    __shared__ int s_n;
    const T* __restrict__ cf = c + (size_t)blockIdx.y * g.N;
    T* __restrict__ kf = kappa + (size_t)blockIdx.y * g.N;
    const int lane = threadIdx.x & 31;
    // (unsigned: a grid's stride past the last cell of 2^31 stays below 2^32)
    for (unsigned start = blockIdx.x * TILE; start < (unsigned)g.N; start += gridDim.x * TILE) {
        const int base = (int)start;
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int end = min(TILE, g.N - base);  // a multiple of VW
#pragma unroll 4
        for (int o = threadIdx.x * VW; o < TILE; o += kCurvThreads * VW) {
            T v[VW];
            uint32_t m = 0;
            if (o < end) {
                ldv<VW>(cf + base + o, v);
#pragma unroll
                for (int e = 0; e < VW; ++e) m |= (interfacial(v[e]) ? 1u : 0u) << e;
                if (FILL) {
#pragma unroll
                    for (int e = 0; e < VW; ++e) v[e] = nan_of<T>();
                    stv<VW>(kf + base + o, v);
                }
            }
            if (__any_sync(0xffffffffu, m != 0u)) {
                int at = warp_reserve(__popc(m), lane, &s_n);
#pragma unroll
                for (int e = 0; e < VW; ++e)
                    if ((m >> e) & 1u) s_cell[at++] = (uint16_t)(o + e);
            }
        }
        __syncthreads();
        const int n = s_n;
        for (int q = threadIdx.x; q < n; q += kCurvThreads) {
            const int x = base + s_cell[q];
            int i, j, k;
            decode(x, g, i, j, k);
            kf[x] = cell_curvature(cf, g, x, i, j, k, h);
        }
        __syncthreads();
    }
}

// f[d][x] on the low d-face of cell x: sum over the K fields of
// gamma kappa_f (c(x) - c(x - e_d)) / h, kappa_f the mean of the two cells'
// curvatures where both have one, else the one that does, else 0.  Only an
// interfacial cell can have a curvature (kappa holds nothing elsewhere).  Faces
// without a curvature add 0 and are left out, except where 0 times the rest is not
// 0: a NaN or an infinity in c reaches the faces beside it.  zero: gamma * 0 / h,
// a NaN for a gamma or h beyond the range of T.  A thread takes VW cells of a row.
template <typename T, int VW>
__global__ void __launch_bounds__(256, 4) k_surface_tension(const T* __restrict__ c, const T* __restrict__ kappa, int K,
                                                         Dims g, T h, T gamma, T zero, T* __restrict__ f) {
    // (one division a thread in FP32 is faster than the parameter held: 157 us
    // against 161 at 192^3 with 7 fields; in double it is a tenth of the pass)
    if constexpr (sizeof(T) == 4) zero = gamma * T(0) / h;
    const bool all_faces = !is_exact_zero(zero);
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < (unsigned)g.N / VW; t += gridDim.x * blockDim.x) {
        const int x = (int)t * VW;
        int i, j, k;
        decode(x, g, i, j, k);
        const int xp = i == 0 ? x + g.nx - 1 : x - 1;  // the cell before the thread's first
        const int ly = j == 0 ? (g.ny - 1) * g.nx : -g.nx;
        const int lz = (k == 0 ? g.nz - 1 : -1) * g.nx * g.ny;
        T acc[3][VW];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int e = 0; e < VW; ++e) acc[d][e] = T(0);
#pragma unroll 2
        for (int q = 0; q < K; ++q) {
            const T* __restrict__ cq = c + (size_t)q * g.N;
            const T* __restrict__ kq = kappa + (size_t)q * g.N;
            T cr[VW], cl[3][VW];
            ldv<VW>(cq + x, cr);
            ldv<VW>(cq + x + ly, cl[1]);
            ldv<VW>(cq + x + lz, cl[2]);
            const T cp = cq[xp];
            std::conditional_t<sizeof(T) == 8, Unsettled64, Unsettled32> u{all_faces};
            u.see(cp);
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                cl[0][e] = e == 0 ? cp : cr[e == 0 ? 0 : e - 1];
                u.see(cr[e]);
                u.see(cl[1][e]);
                u.see(cl[2][e]);
            }
            if (!u.found()) continue;
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                const T kr = interfacial(cr[e]) ? kq[x + e] : nan_of<T>();
                const int xl[3] = {e == 0 ? xp : x + e - 1, x + e + ly, x + e + lz};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const T kl = interfacial(cl[d][e]) ? kq[xl[d]] : nan_of<T>();
                    const bool fl = finite_bits(kl), fr = finite_bits(kr);
                    if (!fl && !fr) {
                        add_nothing(acc[d][e], zero, all_faces, cr[e], cl[d][e]);
                        continue;
                    }
                    const T kf = fl && fr ? T(0.5) * (kl + kr) : (fl ? kl : kr);
                    acc[d][e] += gamma * kf * (cr[e] - cl[d][e]) / h;
                }
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) stv<VW>(f + (size_t)d * g.N + x, acc[d]);
    }
}

// Whole 16-byte lanes on aligned buffers, or a cell at a time.
template <typename T>
static bool whole_lanes(const Dims& g, const void* p, const void* q) {
    return g.nx % VecOf<T>::W == 0 && (((uintptr_t)p | (uintptr_t)q) & 15) == 0;
}

template <typename T, bool FILL, int TILE>
static void curvature_tiles(const T* c, int K, const Dims& g, T h, T* kappa, cudaStream_t st) {
    const dim3 grid(grid_for(g.N, TILE, std::max(1, sm_count() * 32 / K)), K);
    if (whole_lanes<T>(g, c, kappa))
        k_curvature<T, VecOf<T>::W, FILL, TILE><<<grid, kCurvThreads, 0, st>>>(c, g, h, kappa);
    else
        k_curvature<T, 1, FILL, TILE><<<grid, kCurvThreads, 0, st>>>(c, g, h, kappa);
}
// Tiles of fewer cells while they are too few to give every SM four blocks: a
// tile's interfacial cells are a block's serial work (every cell interfacial in
// double: 16^3 took 128 us in tiles of 8192 and takes 19 now, 64^3 246 and 58; drops in
// 28^3 72 and 22).  Half and twice as many blocks: 75 x 90 x 101 takes 17% and 21%
// longer in FP32.
template <typename T, bool FILL>
static void curvature_launch(const T* c, int K, const Dims& g, T h, T* kappa, cudaStream_t st) {
    const long long cells = (long long)g.N * K / (4 * sm_count());
    if (cells >= 8192) curvature_tiles<T, FILL, 8192>(c, K, g, h, kappa, st);
    else if (cells >= 1024) curvature_tiles<T, FILL, 2048>(c, K, g, h, kappa, st);
    else curvature_tiles<T, FILL, 256>(c, K, g, h, kappa, st);
}

template <typename T>
static void tension_launch(const T* c, const T* kappa, int K, const Dims& g, T h, T gamma, T* f, cudaStream_t st) {
    const T zero = gamma * T(0) / h;
    if (whole_lanes<T>(g, c, f))
        k_surface_tension<T, VecOf<T>::W>
            <<<grid_for(g.N / VecOf<T>::W, 256), 256, 0, st>>>(c, kappa, K, g, h, gamma, zero, f);
    else
        k_surface_tension<T, 1><<<grid_for(g.N, 256), 256, 0, st>>>(c, kappa, K, g, h, gamma, zero, f);
}

// Curvatures of K consecutive fields; fill: NaN in every cell without one.
cudaError_t curvature_fields(bool fp64, const void* c, int K, const Dims& g, double h, void* kappa, bool fill,
                             cudaStream_t st) {
    if (K <= 0) return cudaSuccess;
    if (fp64) {
        if (fill) curvature_launch<double, true>((const double*)c, K, g, h, (double*)kappa, st);
        else curvature_launch<double, false>((const double*)c, K, g, h, (double*)kappa, st);
    } else {
        if (fill) curvature_launch<float, true>((const float*)c, K, g, (float)h, (float*)kappa, st);
        else curvature_launch<float, false>((const float*)c, K, g, (float)h, (float*)kappa, st);
    }
    return cudaGetLastError();
}

cudaError_t surface_tension(bool fp64, const void* c, const void* kappa, int K, const Dims& g, double h,
                            double gamma, void* f, cudaStream_t st) {
    if (fp64) tension_launch<double>((const double*)c, (const double*)kappa, K, g, h, gamma, (double*)f, st);
    else tension_launch<float>((const float*)c, (const float*)kappa, K, g, (float)h, (float)gamma, (float*)f, st);
    return cudaGetLastError();
}

}  // namespace vof
