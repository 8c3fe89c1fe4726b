// Step 4 (recolouring) kernels, drop table and nearest-particle statistics
// (Section 2.3 Step 4; Section 3), plus the stateless PLIC primitives.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "plic.cuh"
#include "update_vec.cuh"

namespace vof {

// --------------------------------------------------------------------------
// Step 4

// Occupancy bits of the cells of moving drops, one bit plane per field of
// mv_fields (same row layout as the occupancy bits).  A lane takes a word:
// only its occupied cells (the field's occupancy bits, from which its tags
// were made) read their tag.
__global__ void __launch_bounds__(256) k_moving_bits(const int* __restrict__ labels,
                                                     const uint32_t* __restrict__ bits, Dims g, MoveTables mt,
                                                     const int* __restrict__ mv_fields, int n_mv_fields,
                                                     uint32_t* __restrict__ mvbits) {
    const long long per_field = (long long)g.rows * g.W;
    const long long words = (long long)n_mv_fields * per_field;
    for (long long wd = (long long)blockIdx.x * blockDim.x + threadIdx.x; wd < words;
         wd += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(wd / per_field);
        const int rem = (int)(wd - (long long)q * per_field);
        const int f = mv_fields[q];
        uint32_t occ = bits[(size_t)f * per_field + rem], mv = 0u;
        if (occ) {
            const int row = rem / g.W, wi = rem - row * g.W;
            const int* lab = labels + (size_t)f * g.N + (size_t)row * g.nx + wi * 32;
            while (occ) {
                const int b = __ffs(occ) - 1;
                occ &= occ - 1u;
                const int l = lab[b];
                if (is_moving(mt, f, l)) mv |= 1u << b;
            }
        }
        mvbits[wd] = mv;
    }
}

// 64 consecutive occupancy bits of a row starting at cell x0 (periodic).
__device__ __forceinline__ unsigned long long row_window64(const uint32_t* __restrict__ row, int W, int nx, int x0) {
    return (unsigned long long)row_window(row, W, nx, x0) |
           ((unsigned long long)row_window(row, W, nx, x0 + 32) << 32);
}

// For every moving drop m: the fields (other than its own) with an occupied
// cell within Chebyshev distance `reach` of a cell of m (touch[m], a field
// mask), and the other moving drops within that distance (conflict[m], a
// bit per moving drop).  dil_bits holds the occupancy of every active field
// dilated by `reach`, dil_mv the moving-drop bits dilated the same way.  One
// warp takes one 32-cell word of a moving-drop bit plane at a time and
// groups its set bits by drop.  A group touches field n where n's dilated
// occupancy meets it (lane n tests field n).  Conflicts are searched cell by
// cell only in the moving fields whose dilated bits meet the group (its own
// field always, for the field's other moving drops): the lanes share the
// (2 reach + 1)^2 rows of the window and read each row as a 64-bit window
// (reach <= 16) against the group dilated along x.
__global__ void __launch_bounds__(256) k_touch_words(const int* __restrict__ labels,
                                                     const uint32_t* __restrict__ mvbits,
                                                     const uint32_t* __restrict__ dil_bits,
                                                     const uint32_t* __restrict__ dil_mv, Dims g, int n_active,
                                                     int reach, MoveTables mt, const int* __restrict__ mv_fields,
                                                     int n_mv_fields, unsigned* __restrict__ touch,
                                                     unsigned* __restrict__ conflict, int Mw) {
    const int lane = threadIdx.x & 31;
    const long long per_field = (long long)g.rows * g.W;
    const long long words = (long long)n_mv_fields * per_field;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int span = 2 * reach + 1, nrows = span * span;
    for (long long base = warp * 32; base < words; base += nwarps * 32) {
        // 32 words per round, one per lane; then every non-empty one in turn
        const long long my = base + lane;
        const uint32_t mine = my < words ? mvbits[my] : 0u;
        unsigned todo = __ballot_sync(0xffffffffu, mine != 0u);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1u;
            const long long wd = base + src;
            const uint32_t word = __shfl_sync(0xffffffffu, mine, src);
            const int q = (int)(wd / per_field);
            const long long rem = wd - (long long)q * per_field;
            const int row = (int)(rem / g.W);
            const int wi = (int)(rem - (long long)row * g.W);
            const int j = row % g.ny, k = row / g.ny;
            const int f = mv_fields[q];
            const int* lab = labels + (size_t)f * g.N + (size_t)row * g.nx;
            // the moving drop of each set bit
            const bool set = (word >> lane) & 1u;
            const int m_lane = set ? moving_index(mt, f, lab[wi * 32 + lane]) : -1;
            // this word of every dilated plane, one plane per lane
            const uint32_t db = lane < n_active ? dil_bits[(size_t)lane * per_field + rem] : 0u;
            const uint32_t dm = lane < n_mv_fields ? dil_mv[(size_t)lane * per_field + rem] : 0u;
            unsigned rest = __ballot_sync(0xffffffffu, set);
            while (rest) {
                const int lead = __ffs(rest) - 1;
                const int m = __shfl_sync(0xffffffffu, m_lane, lead);
                const unsigned grp = __ballot_sync(0xffffffffu, set && m_lane == m);
                rest &= ~grp;
                if (m < 0) continue;
                const unsigned tmask = __ballot_sync(0xffffffffu, lane != f && (db & grp) != 0u);
                if (lane == 0 && tmask) atomicOr(touch + m, tmask);
                const unsigned cand = __ballot_sync(0xffffffffu, lane == q || (dm & grp) != 0u);
                // frame bit c <-> cell 32 wi - reach + c; cells within reach
                // along x of the group's cells
                unsigned long long dil = 0;
                for (int s2 = 0; s2 <= 2 * reach; ++s2) dil |= (unsigned long long)grp << s2;
                const int x0 = wi * 32 - reach;
                for (int r2 = lane; r2 < nrows; r2 += 32) {
                    const int dz = r2 / span - reach, dy = r2 % span - reach;
                    const int kk = wrapi(k + dz, g.nz), jj = wrapi(j + dy, g.ny);
                    const size_t roff = (size_t)(kk * g.ny + jj) * g.W;
                    unsigned cm = cand;
                    while (cm) {
                        const int q2 = __ffs(cm) - 1;
                        cm &= cm - 1u;
                        unsigned long long wv = row_window64(mvbits + (size_t)q2 * per_field + roff, g.W, g.nx, x0) & dil;
                        const int f2 = mv_fields[q2];
                        while (wv) {
                            const int b = __ffsll((long long)wv) - 1;
                            wv &= wv - 1ull;
                            const int y = cell(wrapi(x0 + b, g.nx), jj, kk, g);
                            const int l2 = labels[(size_t)f2 * g.N + y];
                            if (f2 == f && l2 == mt.mv_label[m]) continue;  // the drop's own cell
                            const int m2 = moving_index(mt, f2, l2);
                            if (m2 < 0 || m2 == m) continue;
                            const unsigned bitm = 1u << (m2 & 31);
                            unsigned* wd2 = conflict + (size_t)m * Mw + (m2 >> 5);
                            if (!(*wd2 & bitm)) atomicOr(wd2, bitm);
                        }
                    }
                }
            }
        }
    }
}

// dil: workspace of (n_active + 2 * n_mv_fields) bit planes.
cudaError_t recolour_touch(const int* labels, const uint32_t* bits, uint32_t* mvbits, uint32_t* dil, const Dims& g,
                           int n_active, int reach, MoveTables mt, const int* mv_fields, int n_mv_fields,
                           unsigned* touch, unsigned* conflict, int Mw, cudaStream_t st, long long* launches) {
    if (reach > 16) return cudaErrorInvalidValue;  // the 64-cell frame holds 32 + 2 reach cells
    if (n_active > 32 || n_mv_fields > 32) return cudaErrorInvalidValue;  // one lane per plane
    const long long pf = (long long)g.rows * g.W;
    const long long words = (long long)n_mv_fields * pf;
    uint32_t* dil_bits = dil;
    uint32_t* dil_mv = dil + (size_t)n_active * pf;
    uint32_t* tmp = dil_mv + (size_t)n_mv_fields * pf;
    k_moving_bits<<<grid_for(words, 256), 256, 0, st>>>(labels, bits, g, mt, mv_fields, n_mv_fields, mvbits);
    cudaError_t e = dilate_planes(bits, dil_bits, tmp, n_active, g, reach, st);
    if (e == cudaSuccess) e = dilate_planes(mvbits, dil_mv, tmp, n_mv_fields, g, reach, st);
    if (e != cudaSuccess) return e;
    k_touch_words<<<grid_for(words, 256), 256, 0, st>>>(labels, mvbits, dil_bits, dil_mv, g, n_active, reach, mt,
                                                         mv_fields, n_mv_fields, touch, conflict, Mw);
    if (launches) *launches += 8;
    return cudaGetLastError();
}

// Step 4's move: every cell of a moving drop hands its c to the drop's
// target field.  A lane takes a word of the moving-drop bits; only its set
// cells are touched.
template <typename T>
__global__ void __launch_bounds__(256) k_move(T* c, const int* __restrict__ labels,
                                              const uint32_t* __restrict__ mvbits, Dims g, MoveTables mt,
                                              const int* __restrict__ mv_fields, int n_mv_fields,
                                              const int* __restrict__ target, uint32_t* __restrict__ nzc,
                                              uint32_t* __restrict__ nze) {
    const long long per_field = (long long)g.rows * g.W;
    const long long words = (long long)n_mv_fields * per_field;
    for (long long wd = (long long)blockIdx.x * blockDim.x + threadIdx.x; wd < words;
         wd += (long long)gridDim.x * blockDim.x) {
        uint32_t mv = mvbits[wd];
        if (!mv) continue;
        uint32_t filled = 0;
        const int q = (int)(wd / per_field);
        const long long rem = wd - (long long)q * per_field;
        const int row = (int)(rem / g.W), wi = (int)(rem - (long long)row * g.W);
        const int f = mv_fields[q];
        const size_t x0 = (size_t)row * g.nx + wi * 32;
        while (mv) {
            const int b = __ffs(mv) - 1;
            mv &= mv - 1u;
            const size_t x = x0 + b;
            const int m = moving_index(mt, f, labels[(size_t)f * g.N + x]);
            const int tg = m >= 0 ? target[m] : -1;
            if (tg < 0) continue;
            const T v = c[(size_t)f * g.N + x];
            c[(size_t)tg * g.N + x] += v;
            c[(size_t)f * g.N + x] = T(0);
            filled |= 1u << tg;
        }
        if (filled) {
            atomicOr(nzc + (rem >> 1), filled << (16 * (int)(rem & 1)));
            atomicOr(nze + rem, filled * 0x10001u);  // (either end may be among them)
        }
    }
}

// One block per listed field sets the bits of its moving tags.
__global__ void k_move_map(MoveTables mt, uint32_t* __restrict__ map, const int* __restrict__ mv_fields) {
    const int f = mv_fields[blockIdx.x];
    const int lo = mt.mv_start[f], n = mt.mv_count[f];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int l = mt.mv_label[lo + k];
        if (l > 0 && l < kMoveMapTags) atomicOr(map + (size_t)f * kMoveMapWords + (l >> 5), 1u << (l & 31));
    }
}

cudaError_t move_map(MoveTables mt, uint32_t* map, const int* mv_fields, int n_fields, cudaStream_t st) {
    if (n_fields <= 0) return cudaSuccess;
    k_move_map<<<n_fields, 128, 0, st>>>(mt, map, mv_fields);
    return cudaGetLastError();
}

cudaError_t recolour_move(void* c, bool fp64, const int* labels, const uint32_t* mvbits, const Dims& g,
                          MoveTables mt, const int* mv_fields, int n_mv_fields, const int* target, uint16_t* nzc,
                          uint32_t* nze, cudaStream_t st) {
    const long long words = (long long)n_mv_fields * g.rows * g.W;
    uint32_t* nz = reinterpret_cast<uint32_t*>(nzc);
    if (fp64)
        k_move<double><<<grid_for(words, 256), 256, 0, st>>>((double*)c, labels, mvbits, g, mt, mv_fields,
                                                            n_mv_fields, target, nz, nze);
    else
        k_move<float><<<grid_for(words, 256), 256, 0, st>>>((float*)c, labels, mvbits, g, mt, mv_fields,
                                                           n_mv_fields, target, nz, nze);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Drop sums: for every tag the sum of c and its first moments about the tag's
// root (its smallest linear index, minimum image), or the inertia tensor about
// a centre.  Within a row the cells of a tag form runs of few words, and y and
// z are constant on a run, so a run needs only the sums of c, c k and c k^2
// over its cells (k: cells from the run's first) before it adds its share to
// the tag.  FP32 values are summed exactly as 64-bit integers in units
// of 2^-50 (FP64 sums per cell would cost more than everything else: GB300
// issues FP64 at 1/64 of its FP32 rate).
// 256^3, K = 8, phi = 0.3 in FP32 (2347 drops): 0.18 ms for the sums (latency of
// the chain word, label, root) and 0.31 ms for the inertia (FP64 pipe 72%
// busy with the terms of a run); with an atomic per cell and moment they took
// 1.2 and 2.6 ms.  Sums kept over strips of 8 rows, with a fifth of the
// atomics, took 0.8 ms together (fewer warps, their rows in series).

enum DropMode { DropRoots, DropSums, DropInertia };

struct DropOut {
    int* root;            // smallest cell (DropRoots: result, DropSums: input)
    double* S;            // DropSums [4]
    const double* cen;    // DropInertia: centres
    double* I;            // DropInertia [6]
    double h;
};

// Sums of c, c k and c k^2 of a run.
template <typename T>
struct RunSums;
template <>
struct RunSums<double> {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    bool exact = true;  // the sums hold every cell
    __device__ __forceinline__ void add(double v, int k) {
        s0 += v;
        s1 = fma((double)k, v, s1);
        s2 = fma((double)(k * k), v, s2);
    }
    __device__ __forceinline__ double d0() const { return s0; }
    __device__ __forceinline__ double d1() const { return s1; }
    __device__ __forceinline__ double d2() const { return s2; }
};
template <>
struct RunSums<float> {
    unsigned long long s0 = 0, s1 = 0, s2 = 0;  // units of 2^-50; at most 2^50 * 10416 < 2^64
    bool exact = true;
    __device__ __forceinline__ void add(float v, int k) {
        // a float in [2^-26, 1] is a whole number of units; others (none of
        // a step's drops with the default threshold) go cell by cell
        if (!(v == 0.f || (v >= 1.4901161e-8f && v <= 1.f))) exact = false;
        const unsigned long long q = (unsigned long long)(v * 1125899906842624.f);
        s0 += q;
        s1 += q * (unsigned)k;
        s2 += q * (unsigned)(k * k);
    }
    __device__ __forceinline__ double d0() const { return (double)s0 * 8.8817841970012523e-16; }
    __device__ __forceinline__ double d1() const { return (double)s1 * 8.8817841970012523e-16; }
    __device__ __forceinline__ double d2() const { return (double)s2 * 8.8817841970012523e-16; }
};

// Offset t within a period n under the minimum image.
__device__ __forceinline__ int image_offset(int t, int n) {
    if (2 * t >= n) t -= n;
    if (2 * t < -n) t += n;
    return t;
}
// The period to add to t for the minimum image in a box of length L.
__device__ __forceinline__ double image_shift(double t, double L) {
    double s = 0.0;
    if (t > 0.5 * L) s = -L;
    if (t + s < -0.5 * L) s += L;
    return s;
}

// A run of `cnt` cells from (i, j, k) (cell x) whose drop is `idx`: its share
// added to the drop.
template <typename T, DropMode MODE>
__device__ __forceinline__ void add_run(const T* __restrict__ cf, const Dims& g, const DropOut& o, int idx, int x, int i,
                                        int j, int k, int cnt, const RunSums<T>& rs) {
    if (MODE == DropRoots) {
        atomicMin(reinterpret_cast<unsigned*>(o.root) + idx, (unsigned)x);
    } else if (MODE == DropSums) {
        int ri, rj, rk;
        decode(o.root[idx], g, ri, rj, rk);
        const int d1 = image_offset(j - rj, g.ny), d2 = image_offset(k - rk, g.nz);
        const int a = image_offset(i - ri, g.nx), z = image_offset(i + cnt - 1 - ri, g.nx);
        double* s = o.S + 4 * (size_t)idx;
        double s0, s1;
        if (rs.exact && z - a == cnt - 1) {
            s0 = rs.d0();
            s1 = fma((double)a, s0, rs.d1());
        } else {  // the run crosses the half period from the root, or holds a cell the sums do not
            s0 = s1 = 0.0;
            for (int q = 0; q < cnt; ++q) {
                const double v = (double)cf[x + q];
                s0 += v;
                s1 = fma((double)image_offset(i + q - ri, g.nx), v, s1);
            }
        }
        atomicAdd(s + 0, s0);
        atomicAdd(s + 1, s1);
        if (d1) atomicAdd(s + 2, s0 * (double)d1);
        if (d2) atomicAdd(s + 3, s0 * (double)d2);
    } else if (MODE == DropInertia) {
        const double h = o.h, Lx = g.nx * h;
        const double* c = o.cen + 3 * (size_t)idx;
        double r1 = ((double)j + 0.5) * h - c[1], r2 = ((double)k + 0.5) * h - c[2];
        r1 += image_shift(r1, g.ny * h);
        r2 += image_shift(r2, g.nz * h);
        const double ta = ((double)i + 0.5) * h - c[0], tz = ((double)(i + cnt - 1) + 0.5) * h - c[0];
        const double sh = image_shift(ta, Lx);
        double s0, x1, x2;  // sums of c, c t and c t^2, t along x from the centre
        if (rs.exact && sh == image_shift(tz, Lx)) {
            // about the run's middle, so that the terms stay of the run's own size
            const double kc = 0.5 * (double)(cnt - 1), u0 = rs.d0(), u1 = rs.d1(), u2 = rs.d2();
            const double m1 = fma(-kc, u0, u1), m2 = fma(kc * kc, u0, fma(-2.0 * kc, u1, u2));
            const double tc = fma(kc, h, ta + sh);
            s0 = u0;
            x1 = fma(tc, u0, h * m1);
            x2 = fma(tc * tc, u0, fma(2.0 * tc * h, m1, h * h * m2));
        } else {
            s0 = x1 = x2 = 0.0;
            for (int q = 0; q < cnt; ++q) {
                const double v = (double)cf[x + q];
                double t = ((double)(i + q) + 0.5) * h - c[0];
                t += image_shift(t, Lx);
                s0 += v;
                x1 = fma(t, v, x1);
                x2 = fma(t * t, v, x2);
            }
        }
        const double w = h * h * h, own = h * h / 6.0, q1 = r1 * r1, q2 = r2 * r2;
        double* s = o.I + 6 * (size_t)idx;
        atomicAdd(s + 0, w * (s0 * (q1 + q2 + own)));
        atomicAdd(s + 1, w * fma(s0, q2 + own, x2));
        atomicAdd(s + 2, w * fma(s0, q1 + own, x2));
        atomicAdd(s + 3, -w * (x1 * r1));
        atomicAdd(s + 4, -w * (x1 * r2));
        atomicAdd(s + 5, -w * (s0 * (r1 * r2)));
    }
}

// Warps work on their own: a warp collects the occupied words of a tile of
// 32 `rounds` words, stages up to 32 of them in shared memory with coalesced
// loads (all in flight together), and gives each lane one.
constexpr int kDropWarps = 2, kDropRounds = 4;

template <typename T, DropMode MODE, bool BITS>
__global__ void __launch_bounds__(32 * kDropWarps) k_drop_words(const __grid_constant__ DropFields D, Dims g, DropOut o,
                                                                int rounds) {
    __shared__ int s_word[kDropWarps][32 * kDropRounds];
    __shared__ uint32_t s_mask[kDropWarps][32 * kDropRounds];
    __shared__ T s_c[kDropWarps][32][33];                // value of cell b of the lane's word: [b][lane]
    __shared__ int s_lab[kDropWarps][BITS ? 1 : 32][33]; // its tag (BITS: a run's first cell has the tag of all)
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int words = g.rows * g.W;
    const bool whole = (g.nx & 31) == 0;
    const int f = D.ls.f[blockIdx.y];
    int first = 0;  // drops of the slots before this one
    if (D.n_out)
        for (int q = 0; q < (int)blockIdx.y; ++q) first += D.n_out[D.ls.f[q]];
    const int* __restrict__ lab = D.labels + (size_t)f * g.N;
    const T* __restrict__ cf = (const T*)D.c + (size_t)f * g.N;
    // first cell of word w, and the cells it has
    auto place = [&](int w, int& x0, int& cells) {
        if (whole) {
            x0 = w * 32;
            cells = 32;
        } else {
            const int row = w / g.W, i0 = (w - row * g.W) * 32;
            x0 = row * g.nx + i0;
            cells = min(32, g.nx - i0);
        }
    };
    for (int w0 = (blockIdx.x * kDropWarps + wp) * 32 * rounds; w0 < words;
         w0 += gridDim.x * kDropWarps * 32 * rounds) {
        int n = 0;  // occupied words so far, the same on every lane
        for (int r = 0; r < rounds; ++r) {
            const int word = w0 + 32 * r + lane;
            uint32_t m = 0;
            if (BITS) {
                m = word < words ? D.bits[(size_t)f * words + word] : 0u;
            } else {
#pragma unroll 8
                for (int q = 0; q < 32; ++q) {
                    const int w = w0 + 32 * r + q;
                    int x0 = 0, cells = 0;
                    if (w < words) place(w, x0, cells);
                    const unsigned b = __ballot_sync(0xffffffffu, lane < cells && lab[x0 + lane] > 0);
                    if (lane == q) m = b;
                }
            }
            const unsigned vote = __ballot_sync(0xffffffffu, m != 0u);
            if (m) {
                const int at = n + __popc(vote & ((1u << lane) - 1u));
                s_word[wp][at] = word;
                s_mask[wp][at] = m;
            }
            n += __popc(vote);
        }
        __syncwarp();
        for (int base = 0; base < n; base += 32) {
            const int have = min(32, n - base);
#pragma unroll 8
            for (int q = 0; q < have; ++q) {
                int x0, cells;
                place(s_word[wp][base + q], x0, cells);
                if (lane < cells) {
                    if (MODE != DropRoots) s_c[wp][lane][q] = cf[x0 + lane];
                    if (!BITS) s_lab[wp][lane][q] = lab[x0 + lane];
                }
            }
            __syncwarp();
            if (lane < have) {
                const int w = s_word[wp][base + lane];
                uint32_t rest = s_mask[wp][base + lane];
                const int row = w / g.W, i0 = (w - row * g.W) * 32;
                const int j = row % g.ny, k = row / g.ny;
                const int x0 = row * g.nx + i0;
                while (rest) {
                    const int b0 = __ffs(rest) - 1;
                    const int l = BITS ? lab[x0 + b0] : s_lab[wp][b0][lane];
                    RunSums<T> rs;
                    int b = b0;
                    do {  // the run: consecutive cells of one tag
                        if (MODE != DropRoots) rs.add(s_c[wp][b][lane], b - b0);
                        rest &= rest - 1u;
                        ++b;
                    } while (b < 32 && ((rest >> b) & 1u) && (BITS || s_lab[wp][b][lane] == l));
                    if (l > 0 && first + l <= D.n_max)
                        add_run<T, MODE>(cf, g, o, first + l - 1, x0 + b0, i0 + b0, j, k, b - b0, rs);
                }
            }
            __syncwarp();
        }
    }
}

template <DropMode MODE>
static void launch_drop_words(const DropFields& D, const Dims& g, const DropOut& o, cudaStream_t st) {
    // tiles of fewer words while they are too few to give every SM its warps
    const long long words = (long long)g.rows * g.W;
    int rounds = kDropRounds;
    while (rounds > 1 && words * D.ls.n / (32 * rounds) < (long long)sm_count() * 16) rounds /= 2;
    const dim3 grid(grid_for(words, 32 * kDropWarps * rounds, std::max(1, sm_count() * 24 / D.ls.n)), D.ls.n);
    auto go = [&](auto kernel) { kernel<<<grid, 32 * kDropWarps, 0, st>>>(D, g, o, rounds); };
    if constexpr (MODE != DropRoots) {  // (the roots come from labels alone)
        if (D.bits) {
            D.fp64 ? go(k_drop_words<double, MODE, true>) : go(k_drop_words<float, MODE, true>);
            return;
        }
    }
    D.fp64 ? go(k_drop_words<double, MODE, false>) : go(k_drop_words<float, MODE, false>);
}

cudaError_t drop_roots(const DropFields& D, const Dims& g, int* root_of, cudaStream_t st) {
    if (D.n_max <= 0) return cudaSuccess;
    // above every cell's index as an unsigned number
    const cudaError_t e = cudaMemsetAsync(root_of, 0xff, (size_t)D.n_max * 4, st);
    if (e != cudaSuccess) return e;
    launch_drop_words<DropRoots>(D, g, DropOut{root_of, nullptr, nullptr, nullptr, 0.0}, st);
    return cudaGetLastError();
}

cudaError_t drop_sums(const DropFields& D, const Dims& g, const int* root_of, double* S, cudaStream_t st) {
    if (D.n_max <= 0) return cudaSuccess;
    const cudaError_t e = cudaMemsetAsync(S, 0, (size_t)D.n_max * 4 * 8, st);
    if (e != cudaSuccess) return e;
    launch_drop_words<DropSums>(D, g, DropOut{const_cast<int*>(root_of), S, nullptr, nullptr, 0.0}, st);
    return cudaGetLastError();
}

__global__ void k_drop_finalize(const double* __restrict__ S, const int* __restrict__ root_of, Dims g,
                                double h, int n, double* __restrict__ vol, double* __restrict__ cen) {
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        const double* s = S + 4 * (size_t)l;
        int r = root_of[l];
        int rc[3];
        decode(r, g, rc[0], rc[1], rc[2]);
        int L[3] = {g.nx, g.ny, g.nz};
        vol[l] = s[0] * h * h * h;
        for (int a = 0; a < 3; ++a) {
            double p = ((double)rc[a] + 0.5 + s[1 + a] / s[0]) * h;
            double Lh = (double)L[a] * h;
            p = fmod(p, Lh);
            if (p < 0.0) p += Lh;
            if (p >= Lh) p = 0.0;
            cen[3 * (size_t)l + a] = p;
        }
    }
}

cudaError_t drop_finalize(const double* S, const int* root_of, const Dims& g, double h, int n,
                          double* vol, double* cen, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_drop_finalize<<<grid_for(n, 128), 128, 0, st>>>(S, root_of, g, h, n, vol, cen);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Drop shape (Appendix A): inertia tensor of each drop about its centre of
// mass, I = integral over the drop of [(r.r) delta - r r], of the drop's
// colour density (each cell of the tag holding c uniformly: the cell-centre
// term plus the cube's own moment c h^5 / 6 on the diagonal), r under the
// minimum image; and the aspect ratio chi = sqrt(I_max / I_min).

cudaError_t drop_inertia(const DropFields& D, const Dims& g, double h, const double* cen, double* I, cudaStream_t st) {
    if (D.n_max <= 0) return cudaSuccess;
    const cudaError_t e = cudaMemsetAsync(I, 0, (size_t)D.n_max * 6 * 8, st);
    if (e != cudaSuccess) return e;
    launch_drop_words<DropInertia>(D, g, DropOut{nullptr, nullptr, cen, I, h}, st);
    return cudaGetLastError();
}

// Extreme eigenvalues of the symmetric matrix [[a, d, e], [d, b, f], [e, f, c]]:
// with q = tr/3 and B = (A - q 1)/p, p^2 = tr((A - q 1)^2)/6, the eigenvalues
// are q + 2 p cos(phi + 2 pi m / 3), m = 0, 1, 2, where cos(3 phi) = det(B)/2
// (the characteristic polynomial of B is the triple-angle identity).
__device__ __forceinline__ void sym3_extremes(double a, double b, double c, double d, double e, double f,
                                              double& lmax, double& lmin) {
    const double off = d * d + e * e + f * f;
    const double q = (a + b + c) / 3.0;
    const double p2 = ((a - q) * (a - q) + (b - q) * (b - q) + (c - q) * (c - q) + 2.0 * off) / 6.0;
    if (!(p2 > 0.0)) {
        lmax = lmin = q;
        return;
    }
    const double p = sqrt(p2);
    const double B00 = (a - q) / p, B11 = (b - q) / p, B22 = (c - q) / p;
    const double B01 = d / p, B02 = e / p, B12 = f / p;
    const double det = B00 * (B11 * B22 - B12 * B12) - B01 * (B01 * B22 - B12 * B02) + B02 * (B01 * B12 - B11 * B02);
    const double r = fmin(1.0, fmax(-1.0, 0.5 * det));
    const double phi = acos(r) / 3.0;
    lmax = q + 2.0 * p * cos(phi);
    lmin = q + 2.0 * p * cos(phi + 2.0 * M_PI / 3.0);
}

// chi of every drop; acc[0] += sum of chi, acc[1] += drops, acc[2] = max chi.
__global__ void __launch_bounds__(128) k_drop_chi(const double* __restrict__ I, int n, double* __restrict__ chi,
                                                  double* __restrict__ acc) {
    double sum = 0.0, cnt = 0.0, mx = 0.0;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        const double* s = I + 6 * (size_t)l;
        double lmax, lmin;
        sym3_extremes(s[0], s[1], s[2], s[3], s[4], s[5], lmax, lmin);
        const double x = lmin > 0.0 ? sqrt(lmax / lmin) : INFINITY;
        if (chi) chi[l] = x;
        if (isfinite(x)) {
            sum += x;
            cnt += 1.0;
            mx = fmax(mx, x);
        }
    }
    if (!acc) return;
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_down_sync(0xffffffffu, sum, o);
        cnt += __shfl_down_sync(0xffffffffu, cnt, o);
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0 && cnt > 0.0) {
        atomicAdd(acc + 0, sum);
        atomicAdd(acc + 1, cnt);
        // positive doubles order like their bit patterns
        atomicMax(reinterpret_cast<unsigned long long*>(acc + 2), (unsigned long long)__double_as_longlong(mx));
    }
}

cudaError_t drop_chi(const double* I, int n, double* chi, double* acc, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_drop_chi<<<grid_for(n, 128, 1024), 128, 0, st>>>(I, n, chi, acc);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Nearest-particle statistics (Section 3, eq. P_nstij with h_ij = 1/N_i for
// the N_i equidistant nearest neighbours; histograms of eqs. vec_cond and
// Ptheta_r; moments M and R of Section 4).

__device__ __forceinline__ double min_image(double t, double L) {
    if (t > 0.5 * L) t -= L;
    if (t < -0.5 * L) t += L;
    return t;
}

// A warp takes a drop.  Every pair is first measured in FP32 from centroids
// staged in shared memory; only the pairs that may be nearest -- within the
// FP32 minimum plus the tie tolerance plus a bound on the FP32 error -- are
// measured in FP64, usually one or two per drop, from a list per warp.  2347
// drops: 0.06 ms, the FP64 pipe 63% busy with the conversions; a thread per
// drop and three FP64 passes over all pairs took 8.5 ms on 19 blocks.
//
// The bound: converting both coordinates, their difference and the image
// shift round by at most 2^-24 of 6 max(|coordinate|, box) in all, a distance
// by sqrt(3) times that plus a few 2^-24 of itself; `margin` is over three
// times twice this.  Coordinates, boxes or tolerances that overflow FP32 make
// every pair a candidate, and a list that overflows makes the warp measure
// every pair in FP64.
constexpr int kPairTile = 512, kPairWarps = 8, kPairCand = 64;

__global__ void __launch_bounds__(32 * kPairWarps) k_pair_stats(const double* __restrict__ cen, long long n, double bx,
                                                                double by, double bz, int vaxis, int n_rbins, double dr,
                                                                int n_tbins, double dtheta, double tie_tol,
                                                                double* __restrict__ hist_r,
                                                                double* __restrict__ hist_rt,
                                                                double* __restrict__ moments) {
    __shared__ float s_c[3][kPairTile];
    __shared__ long long s_cand[kPairWarps][kPairCand];
    __shared__ double red[13][kPairWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double loc[13];
#pragma unroll
    for (int q = 0; q < 13; ++q) loc[q] = 0.0;
    const float L0 = (float)bx, L1 = (float)by, L2 = (float)bz;
    const float H0 = 0.5f * L0, H1 = 0.5f * L1, H2 = 0.5f * L2;
    auto image = [](float t, float L, float H) {
        if (t > H) t -= L;
        if (t < -H) t += L;
        return t;
    };
    for (long long i0 = (long long)blockIdx.x * kPairWarps; i0 < n; i0 += (long long)gridDim.x * kPairWarps) {
        const long long i = i0 + wid;
        const bool mine = i < n;
        double ci[3] = {0.0, 0.0, 0.0};
        if (mine)
            for (int a = 0; a < 3; ++a) ci[a] = cen[3 * i + a];
        const float f0 = (float)ci[0], f1 = (float)ci[1], f2 = (float)ci[2];
        float best = INFINITY, big = 0.f, thr = 0.f;
        int ncand = 0;  // the same on every lane
        for (int pass = 0; pass < 2; ++pass) {
            for (long long j0 = 0; j0 < n; j0 += kPairTile) {
                const int m = (int)(n - j0 < kPairTile ? n - j0 : kPairTile);
                __syncthreads();
                for (int q = threadIdx.x; q < 3 * m; q += 32 * kPairWarps) s_c[q % 3][q / 3] = (float)cen[3 * j0 + q];
                __syncthreads();
                if (!mine) continue;
                for (int q0 = 0; q0 < m; q0 += 32) {
                    const int q = q0 + lane;
                    const bool on = q < m && j0 + q != i;
                    float d2 = INFINITY;
                    if (on) {
                        const float x = s_c[0][q], y = s_c[1][q], z = s_c[2][q];
                        const float tx = image(x - f0, L0, H0), ty = image(y - f1, L1, H1), tz = image(z - f2, L2, H2);
                        d2 = tx * tx + ty * ty + tz * tz;
                        if (pass == 0) big = fmaxf(big, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
                    }
                    if (pass == 0) {
                        best = fminf(best, d2);
                    } else {
                        const unsigned c = __ballot_sync(0xffffffffu, on && d2 <= thr);
                        if (c) {
                            const int at = ncand + __popc(c & ((1u << lane) - 1u));
                            if (((c >> lane) & 1u) && at < kPairCand) s_cand[wid][at] = j0 + q;
                            ncand += __popc(c);
                        }
                    }
                }
            }
            if (pass == 0) {
                for (int o = 16; o > 0; o >>= 1) {
                    best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
                    big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
                }
                big = fmaxf(big, fmaxf(fabsf(f0), fmaxf(fabsf(f1), fabsf(f2))));
                const float margin = 4e-6f * (L0 + L1 + L2 + big);
                const float t = sqrtf(best) + (float)tie_tol * 1.000001f + margin;
                thr = t * t * 1.000001f;
            }
        }
        __syncwarp();
        if (!mine) continue;
        // FP64 on the candidates (on every drop if they did not fit)
        const bool fits = ncand <= kPairCand;
        const long long nc = fits ? ncand : n;
        auto measure = [&](long long q, double r[3]) {  // distance to candidate q, NaN (never chosen) for the drop itself
            const long long j = fits ? s_cand[wid][q] : q;
            if (j == i) return (double)NAN;
            r[0] = min_image(cen[3 * j] - ci[0], bx);
            r[1] = min_image(cen[3 * j + 1] - ci[1], by);
            r[2] = min_image(cen[3 * j + 2] - ci[2], bz);
            return sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
        };
        double r[3], dmin = INFINITY;
        for (long long q = lane; q < nc; q += 32) {
            const double dd = measure(q, r);
            if (dd < dmin) dmin = dd;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double t = __shfl_xor_sync(0xffffffffu, dmin, o);
            if (t < dmin) dmin = t;
        }
        int ni = 0;
        for (long long q = lane; q < nc; q += 32) ni += measure(q, r) - dmin <= tie_tol ? 1 : 0;
        ni = __reduce_add_sync(0xffffffffu, ni);
        const double wgt = 1.0 / (double)ni;
        for (long long q = lane; q < nc; q += 32) {
            const double dd = measure(q, r);
            if (!(dd - dmin <= tie_tol)) continue;
            int kr = (int)floor(dd / dr);
            if (kr > n_rbins || kr < 0) kr = n_rbins;
            double ct = dd > 0.0 ? r[vaxis] / dd : 1.0;
            if (ct > 1.0) ct = 1.0;
            if (ct < -1.0) ct = -1.0;
            int kt = (int)floor(acos(ct) / dtheta);
            if (kt >= n_tbins) kt = n_tbins - 1;
            if (kt < 0) kt = 0;
            atomicAdd(hist_r + kr, wgt);
            atomicAdd(hist_rt + (size_t)kr * n_tbins + kt, wgt);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                loc[a] += wgt * r[a];
#pragma unroll
                for (int b = 0; b < 3; ++b) loc[3 + 3 * a + b] += wgt * r[a] * r[b];
            }
        }
        if (lane == 0) loc[12] += 1.0;
    }
    // block reduction of the 13 sums
#pragma unroll
    for (int q = 0; q < 13; ++q) {
        double v = loc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[q][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < 13) {
        double v = 0.0;
        for (int w = 0; w < kPairWarps; ++w) v += red[threadIdx.x][w];
        if (v != 0.0) atomicAdd(moments + threadIdx.x, v);
    }
}

cudaError_t pair_stats(const double* cen, long long n, double bx, double by, double bz, int vaxis,
                       int n_rbins, double dr, int n_tbins, double dtheta, double tie_tol, double* hist_r,
                       double* hist_rt, double* moments, cudaStream_t st) {
    if (n < 2) return cudaSuccess;
    k_pair_stats<<<grid_for(n, kPairWarps), 32 * kPairWarps, 0, st>>>(cen, n, bx, by, bz, vaxis, n_rbins, dr, n_tbins,
                                                                       dtheta, tie_tol, hist_r, hist_rt, moments);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// PLIC primitives, normals, velocity scan

template <typename T>
__global__ void k_plic_volume(const T* __restrict__ m, const T* __restrict__ alpha, T* __restrict__ v,
                              long long n) {
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        v[t] = plic_volume<T>(m[3 * t], m[3 * t + 1], m[3 * t + 2], alpha[t]);
}

template <typename T>
__global__ void k_plic_alpha(const T* __restrict__ m, const T* __restrict__ c, T* __restrict__ alpha,
                             long long n, T band) {
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        alpha[t] = plic_alpha_banded(m[3 * t], m[3 * t + 1], m[3 * t + 2], c[t], band);
}

cudaError_t plic_volume_batch(bool fp64, const void* m, const void* alpha, void* v, long long n,
                              cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (fp64)
        k_plic_volume<double><<<grid_for(n, 128), 128, 0, st>>>((const double*)m, (const double*)alpha,
                                                               (double*)v, n);
    else
        k_plic_volume<float><<<grid_for(n, 128), 128, 0, st>>>((const float*)m, (const float*)alpha,
                                                              (float*)v, n);
    return cudaGetLastError();
}

cudaError_t plic_alpha_batch(bool fp64, const void* m, const void* c, void* alpha, long long n,
                             double band, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (fp64)
        k_plic_alpha<double><<<grid_for(n, 128), 128, 0, st>>>((const double*)m, (const double*)c,
                                                              (double*)alpha, n, band);
    else
        k_plic_alpha<float><<<grid_for(n, 128), 128, 0, st>>>((const float*)m, (const float*)c,
                                                             (float*)alpha, n, (float)band);
    return cudaGetLastError();
}

template <typename T>
__global__ void k_normals(const T* __restrict__ cf, Dims g, T* __restrict__ m) {
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < g.N; x += gridDim.x * blockDim.x) {
        T r[3] = {T(0), T(0), T(0)};
        if (vclass(cf[x]) == 1) {
            int i, j, k;
            decode(x, g, i, j, k);
            T st[27];
            int is[3] = {wrapi(i - 1, g.nx), i, wrapi(i + 1, g.nx)};
            int js[3] = {wrapi(j - 1, g.ny), j, wrapi(j + 1, g.ny)};
            int ks[3] = {wrapi(k - 1, g.nz), k, wrapi(k + 1, g.nz)};
            for (int c = 0; c < 3; ++c)
                for (int b = 0; b < 3; ++b)
                    for (int a = 0; a < 3; ++a) st[c * 9 + b * 3 + a] = cf[cell(is[a], js[b], ks[c], g)];
            myc_normal(st, r);
        }
        m[3 * (size_t)x] = r[0];
        m[3 * (size_t)x + 1] = r[1];
        m[3 * (size_t)x + 2] = r[2];
    }
}

cudaError_t normals_field(bool fp64, const void* cf, const Dims& g, void* m, cudaStream_t st) {
    if (fp64)
        k_normals<double><<<grid_for(g.N, 128), 128, 0, st>>>((const double*)cf, g, (double*)m);
    else
        k_normals<float><<<grid_for(g.N, 128), 128, 0, st>>>((const float*)cf, g, (float*)m);
    return cudaGetLastError();
}

// out[0] = max |u| over the finite values, out[1] = 1 if any is not finite (both
// zero before; the maximum as a double's bits).  Magnitudes order as their bit
// patterns, so the pass runs on integers, 16 bytes a load where u allows it, and
// a block adds one atomic: with one per warp the atomics on one address were
// the time (32 boxes of 32^3 to 128^3 in turn: 0.63 -> 0.14 ms).
template <typename T, typename I>
__global__ void __launch_bounds__(256) k_vscan(const T* __restrict__ u, long long n, long long n_vec,
                                               unsigned long long* __restrict__ out) {
    constexpr I kMag = (I)~(I)0 >> 1, kInf = sizeof(T) == 8 ? (I)0x7ff0000000000000ULL : (I)0x7f800000U;
    constexpr int W = 16 / sizeof(T);
    __shared__ I s_mx[8];
    __shared__ unsigned s_bad;
    I mx = 0;
    unsigned bad = 0;
    auto take = [&](T v) {
        I b;
        memcpy(&b, &v, sizeof(T));
        b &= kMag;
        if (b >= kInf) bad = 1;
        else mx = b > mx ? b : mx;
    };
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
    for (long long t = first; t < n_vec; t += stride) {
        T v[W];
        ldv<W>(u + t * W, v);
#pragma unroll
        for (int e = 0; e < W; ++e) take(v[e]);
    }
    for (long long t = n_vec * W + first; t < n; t += stride) take(u[t]);
    if (threadIdx.x == 0) s_bad = 0u;
    for (int o = 16; o > 0; o >>= 1) {
        const I other = __shfl_down_sync(0xffffffffu, mx, o);
        mx = other > mx ? other : mx;
    }
    if ((threadIdx.x & 31) == 0) s_mx[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&s_bad, 1u);
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; ++w) mx = s_mx[w] > mx ? s_mx[w] : mx;
    T v;
    memcpy(&v, &mx, sizeof(T));
    if (mx != 0) atomicMax(out, (unsigned long long)__double_as_longlong((double)v));
    if (s_bad) atomicOr(out + 1, 1ull);
}

cudaError_t velocity_scan(bool fp64, const void* u, long long n, double* out2, cudaStream_t st) {
    const bool vec = ((uintptr_t)u & 15) == 0;
    const long long n_vec = vec ? n / (fp64 ? 2 : 4) : 0;
    // a few loads a thread: enough blocks for the memory, few atomics
    const int blocks = (int)std::max(1ll, std::min<long long>(sm_count() * 8, (n + 2047) / 2048));
    if (fp64)
        k_vscan<double, unsigned long long>
            <<<blocks, 256, 0, st>>>((const double*)u, n, n_vec, (unsigned long long*)out2);
    else
        k_vscan<float, unsigned><<<blocks, 256, 0, st>>>((const float*)u, n, n_vec, (unsigned long long*)out2);
    return cudaGetLastError();
}

namespace {
thread_local const char* g_last_cuda_error = "no error";
}

cudaError_t note_cuda_error(cudaError_t e) {
    if (e != cudaSuccess) g_last_cuda_error = cudaGetErrorName(e);
    return e;
}

const char* last_cuda_error_name() { return g_last_cuda_error; }

}  // namespace vof
