// Split advection over a set of independent boxes (one box for a context,
// up to kMaxBoxes for a batch): every pass of a sweep is one launch that
// covers every field of every box.
//
// The set travels by value as a __grid_constant__ kernel parameter (10.8 KB
// for 64 boxes in FP32, 11.3 KB in double; read in place from the parameter
// space), so a captured CUDA graph holds it and no table has to be copied to
// the device.
//
// The sweep passes work on words: 32 consecutive cells of a row of one field
// (the unit of the occupancy bits), VW cells per lane and 32 / VW lanes per
// word.  Drops fill a small part of every field, so each buffer that holds a
// state (c and the two scratch buffers) has a map of the words that may hold
// a non-zero value (a bit per field, 16 bits per word of the grid); the
// update pass touches only the words whose result can differ from what its
// output buffer holds.  A tile of up to kTileWords words of one box is the
// unit of work of a block, which lists the tile's active (word, field) items
// in shared memory and hands them to its lane groups.
// The face list of the next sweep holds 64-bit keys (face_key).
#pragma once

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "plic.cuh"
#include "faces.cuh"
#include "update_vec.cuh"

namespace vof {

// Division by a fixed positive divisor d through a multiply-high (the
// round-up method of Granlund & Montgomery 1994), exact for n < 2^31: with
// 2^(l-1) < d < 2^l, mul = ceil(2^(31+l) / d) < 2^32 and
// q = umulhi(n, mul) >> (l - 1); a power of two is a shift.
struct FastDiv {
    uint32_t mul, sh;  // mul == 0: q = n >> sh
};
__host__ inline FastDiv fastdiv_make(uint32_t d) {
    FastDiv f;
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    if ((1ull << l) == d) {
        f.mul = 0;
        f.sh = l;
    } else {
        f.mul = (uint32_t)(((1ull << (31 + l)) + d - 1) / d);
        f.sh = l - 1;
    }
    return f;
}
__device__ __forceinline__ uint32_t fastdiv(uint32_t n, const FastDiv& f) {
    return f.mul == 0 ? (n >> f.sh) : (__umulhi(n, f.mul) >> f.sh);
}

template <typename T>
struct BoxDev {
    Dims g;
    int K;      // fields advected
    int tile0;  // first tile of the box
    int words;  // 32-cell words of one field, rows * W
    FastDiv divW, divnx, divny;  // by W, nx and ny
    T sfac;     // dt / h
    T* c;       // [K][N] state (updated in place over a step)
    T* b1;      // [K][N] state after the first sweep
    T* b2;      // [K][N] state after the second sweep
    T* flux;    // [K][N] flux of listed faces, at the face's high-side cell
    const T* u; // [3][N] face velocities (low faces)
    float4* net;        // [K][N] network normal at listed faces (learned path)
    uint32_t* ccbits;   // [K][rows][W] c > 1/2 at the step start
    uint32_t* occbits;  // [K][rows][W] c > tau after the step
    uint16_t* nzc;      // [rows][W] fields with a non-zero value in the word of c, of b1 and of b2
    uint16_t* nz1;      // (a set bit may stand for a word of zeros)
    uint16_t* nz2;
    uint32_t* nze;      // [rows][W] fields non-zero in the word's first cell (low half) and last cell (high half)
                        // of the state that the next sweep along x reads
    double* clipped;    // [K] volume removed by the clip
};

// NB = capacity: 1 for a context, kMaxBoxes for a batch.
template <typename T, int NB>
struct BoxSet {
    int n;
    int tiles;  // over every box
    int tw;     // words per tile, at most kTileWords
    BoxDev<T> b[NB];
};

static_assert(sizeof(BoxSet<double, kMaxBoxes>) <= 16 * 1024, "well within the 32 KB of kernel parameters");

template <typename T, int NB>
__device__ __forceinline__ int box_of_tile(const BoxSet<T, NB>& S, int tile) {
    if (NB == 1) return 0;
    int lo = 0, hi = S.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (S.b[mid].tile0 <= tile) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename T>
__device__ __forceinline__ const T* sweep_in(const BoxDev<T>& B, int sweep) {
    return sweep == 0 ? B.c : (sweep == 1 ? B.b1 : B.b2);
}
template <typename T>
__device__ __forceinline__ T* sweep_out(const BoxDev<T>& B, int sweep) {
    return sweep == 0 ? B.b1 : (sweep == 1 ? B.b2 : B.c);
}

template <typename T>
__device__ __forceinline__ uint16_t* nz_in(const BoxDev<T>& B, int sweep) {
    return sweep == 0 ? B.nzc : (sweep == 1 ? B.nz1 : B.nz2);
}
template <typename T>
__device__ __forceinline__ uint16_t* nz_out(const BoxDev<T>& B, int sweep) {
    return sweep == 0 ? B.nz1 : (sweep == 1 ? B.nz2 : B.nzc);
}

// Words of a tile: most, and the number for a set of `words` words in all --
// smaller tiles until there are eight to an SM, twice what it holds at once.
constexpr int kTileWords = 128;
constexpr int kSweepThreads = 256;
inline int tile_words(long long words) {
    int tw = kTileWords;
    while (tw > 16 && words / tw < 8 * sm_count()) tw /= 2;
    return tw;
}

// A donor that is not empty.  An FP32 NaN counts as interfacial where a lane
// takes one cell (rows that are not whole lanes), and spreads with the flux; where
// it takes several it counts as empty, and stays in its cell.
template <int VW, typename T>
__device__ __forceinline__ bool holds(T v) {
    return VW == 1 ? vclass(v) != 0 : above_zero(v);
}

// Place of one word of a tile.
struct WordPlace {
    int x0, i0;               // first cell: index in the field, and along x
    int lo, hi;               // offsets of the neighbour rows along d (d != 0)
    int hin;                  // offset of the high neighbour row along dn (dn != 0)
};

// Place of word `word` of a box, with its neighbour words along d.
template <typename T>
__device__ __forceinline__ WordPlace place_word(const BoxDev<T>& B, int word, int d, int dn, int& wlo, int& whi) {
    const Dims& g = B.g;
    WordPlace p;
    const int row = (int)fastdiv((uint32_t)word, B.divW), wi = word - row * g.W;
    const int k = (int)fastdiv((uint32_t)row, B.divny), j = row - k * g.ny;
    p.i0 = wi * 32;
    p.x0 = row * g.nx + p.i0;
    // rows up and down along y and z
    const int ylo = j == 0 ? g.ny - 1 : -1, yhi = j == g.ny - 1 ? 1 - g.ny : 1;
    const int zlo = (k == 0 ? g.nz - 1 : -1) * g.ny, zhi = (k == g.nz - 1 ? 1 - g.nz : 1) * g.ny;
    const int rlo = d == 1 ? ylo : zlo, rhi = d == 1 ? yhi : zhi;
    p.lo = rlo * g.nx;
    p.hi = rhi * g.nx;
    wlo = d == 0 ? word + (wi == 0 ? g.W - 1 : -1) : word + rlo * g.W;
    whi = d == 0 ? word + (wi == g.W - 1 ? 1 - g.W : 1) : word + rhi * g.W;
    p.hin = (dn == 1 ? yhi : zhi) * g.nx;
    return p;
}

// The sweep buffers of every box before the first step, whatever the memory
// held: the active fields zero, and the maps say so (fields past K keep their
// bits: they become active with whatever they hold).  Bound: HBM writes, 2 es
// bytes per cell-field.  Leaving the buffers as they are and every bit of their
// maps set made the first step's first two sweeps touch every word of every
// field (256^3, K = 8: 7.8 ms for a context's
// first FP64 step against 5.2 for the next; now 5.2.  A 32-box FP32 batch with
// its four steps: 9.45 -> 8.94 ms).
template <typename T, int NB>
__global__ void __launch_bounds__(kSweepThreads) k_clear_sp(const __grid_constant__ BoxSet<T, NB> S) {
    for (int tile = blockIdx.x; tile < S.tiles; tile += gridDim.x) {
        const int bx = box_of_tile(S, tile);
        const BoxDev<T>& B = S.b[bx];
        const int lt = tile - B.tile0, tiles = (B.words + S.tw - 1) / S.tw;
        // the tile's share of the fields' 16-byte units (the last one may reach
        // into the padding of the buffer or a field that is not active)
        const long long units = ((long long)B.K * B.g.N * (int)sizeof(T) + 15) / 16, share = (units + tiles - 1) / tiles;
        const long long end = min((lt + 1) * share, units);
        uint4* const b1 = reinterpret_cast<uint4*>(B.b1);
        uint4* const b2 = reinterpret_cast<uint4*>(B.b2);
        for (long long q = lt * share + threadIdx.x; q < end; q += kSweepThreads) {
            b1[q] = make_uint4(0, 0, 0, 0);
            b2[q] = make_uint4(0, 0, 0, 0);
        }
        const uint16_t past = (uint16_t)~((1u << B.K) - 1u);
        const int w = lt * S.tw + (int)threadIdx.x;
        if ((int)threadIdx.x < S.tw && w < B.words) {
            B.nz1[w] = past;
            B.nz2[w] = past;
        }
    }
}

// Faces of sweep d whose upwind donor is interfacial, from the state c of
// every box (start of a call, or after a field was activated), with what the
// update pass keeps up from there on: the map of c's non-zero words and the
// occupancy bits.  A lane group takes a word of every field in turn (the
// velocity read once, four fields' loads in flight).
template <typename T, int NB, int VW>
__global__ void __launch_bounds__(kSweepThreads) k_list_sp(const __grid_constant__ BoxSet<T, NB> S, int d, T tau,
                                                           unsigned long long* __restrict__ list,
                                                           int* __restrict__ count) {
    constexpr int LPW = 32 / VW, WPW = 32 / LPW;  // lanes per word, words per warp
    constexpr int FB = 4;                         // fields in flight
    __shared__ unsigned long long s_buf[kSweepThreads / 32][kWarpBuf];
    const int lane = threadIdx.x & 31, gl = lane & (LPW - 1);
    FaceWriter out(s_buf[threadIdx.x >> 5], list, count);
    const unsigned group = (0xffffffffu >> (32 - LPW)) << (lane & ~(LPW - 1));
    for (int tile = blockIdx.x; tile < S.tiles; tile += gridDim.x) {
        const int bx = box_of_tile(S, tile);
        const BoxDev<T>& B = S.b[bx];
        const Dims& g = B.g;
        const int w0 = (tile - B.tile0) * S.tw, w1 = min(w0 + S.tw, B.words);
        for (int base = w0 + (threadIdx.x >> 5) * WPW; base < w1; base += (kSweepThreads / 32) * WPW) {
            const int word = base + lane / LPW;
            const bool ok = word < w1;
            int wlo, whi;
            const WordPlace p = place_word(B, ok ? word : w0, d, d, wlo, whi);
            const bool valid = ok && p.i0 + gl * VW < g.nx;
            const int i = p.i0 + (valid ? gl * VW : 0), x = p.x0 + (valid ? gl * VW : 0);
            // faces of this lane's cells as donors: the low one where the
            // velocity is negative, the high one where it is positive
            uint32_t nlo = 0, nhi = 0;
            {
                T ul[VW], uh[VW];
                const T* __restrict__ ud = B.u + (size_t)d * g.N;
                ldv<VW>(ud + x, ul);
                if (d == 0) {
                    const T next = next_along_x<T, VW>(ul, ud, x, i, g.nx, gl, LPW);
#pragma unroll
                    for (int e = 0; e < VW; ++e) uh[e] = e == VW - 1 ? next : ul[e + 1];
                } else {
                    ldv<VW>(ud + x + p.hi, uh);
                }
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    nlo |= (valid && vsign(ul[e]) < 0 ? 1u : 0u) << e;
                    nhi |= (valid && vsign(uh[e]) > 0 ? 1u : 0u) << e;
                }
            }
            uint32_t nz = 0, edge_lo = 0, edge_hi = 0;  // fields non-zero in the word, in the lane's first and last cell
            for (int f0 = 0; f0 < B.K; f0 += FB) {
                T cv[FB][VW];
#pragma unroll
                for (int q = 0; q < FB; ++q)
                    if (f0 + q < B.K) ldv<VW>(B.c + (size_t)(f0 + q) * g.N + x, cv[q]);
#pragma unroll
                for (int q = 0; q < FB; ++q) {
                    const int f = f0 + q;
                    if (f >= B.K) break;
                    bool any = false;
                    uint32_t inter = 0, occ = 0;
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        any |= !is_exact_zero(cv[q][e]);
                        inter |= (holds<VW>(cv[q][e]) && !at_least_one(cv[q][e]) ? 1u : 0u) << e;
                        occ |= (above(cv[q][e], tau) ? 1u : 0u) << e;
                    }
                    const unsigned vote = __ballot_sync(0xffffffffu, valid && any);
                    uint32_t ow = 0;
                    if (vote) {  // the same for the warp
                        if (vote & group) nz |= 1u << f;
                        if (d == 0) {
                            edge_lo |= (is_exact_zero(cv[q][0]) ? 0u : 1u) << f;
                            edge_hi |= (is_exact_zero(cv[q][VW - 1]) ? 0u : 1u) << f;
                        }
                        ow = gather_word<VW>(valid ? occ : 0u, lane);
                        const uint32_t fl = inter & nlo, fh = inter & nhi;
                        const int n = __popc(fl) + __popc(fh);
                        if (__any_sync(0xffffffffu, n != 0)) {
                            int pos = out.reserve(n, lane);
#pragma unroll
                            for (int e = 0; e < VW; ++e) {
                                if ((fl >> e) & 1u) out.buf[pos++] = face_key(bx, f, 0, x + e);
                                if ((fh >> e) & 1u) out.buf[pos++] = face_key(bx, f, 1, x + e);
                            }
                            out.settle(lane);
                        }
                    }
                    if (ok && gl == 0) B.occbits[(size_t)f * B.words + word] = ow;
                }
            }
            if (ok && gl == 0) B.nzc[word] = (uint16_t)nz;
            if (d == 0 && valid) {
                uint16_t* const e16 = reinterpret_cast<uint16_t*>(B.nze + word);
                if (gl == 0) e16[0] = (uint16_t)edge_lo;
                if (i + VW == min(p.i0 + 32, g.nx)) e16[1] = (uint16_t)edge_hi;
            }
        }
    }
    out.flush(lane);
}

// Update pass of sweep PH (0, 1, 2) along d (DX: d == 0) for every box:
// c_out = c_in - (F_hi - F_lo) + c_c (s_hi - s_lo), c_c bits written in
// sweep 0 and read after, the clip and the occupancy bits in sweep 2, and the
// faces of the next sweep (direction dn) whose donor is interfacial appended
// to its list.
//
// A word of a field is active when it, or a neighbour word along d, may be
// non-zero in the input, or when the output buffer may hold something there
// that has to become zero; every other word is zero in both buffers and is
// neither read nor written (drops fill a few per cent of a field: one word in
// five is active at phi = 0.3 in 8 fields).  Along x a neighbour word counts by
// its cell next to this one alone: the pass (or listing) before a sweep along x
// leaves a map of the words' end cells (whole neighbour words made the sweep take
// 1.7 times as long).  The block collects the tile's
// active (word, field) items in shared memory, so that lane groups work on
// full items whatever their pattern; items of a word follow each other, so
// its velocities come from L1 after the first.
//
// Bound: latency (three dependent loads per item: map, values, listed flux).
// 256^3, K = 8, phi = 0.3, FP32: 0.17 ms per y or z sweep (0.38 ms when every
// word of every field was read and written), 0.16 ms per x sweep (0.43 ms; 0.28 ms
// with whole neighbour words); FP64 0.68 to 0.79 ms.
template <typename T, int NB, int VW, int PH, bool DX>
__global__ void __launch_bounds__(kSweepThreads, 4)
    k_update_sp(const __grid_constant__ BoxSet<T, NB> S, int d, int dn, T tau,
                unsigned long long* __restrict__ nlist, int* __restrict__ ncount) {
    constexpr int LPW = 32 / VW, WPW = 32 / LPW;
    constexpr int WARPS = kSweepThreads / 32;
    __shared__ unsigned long long s_buf[WARPS][kWarpBuf];
    __shared__ int s_warp[WARPS];
    __shared__ WordPlace s_place[kTileWords];
    __shared__ uint16_t s_item[kTileWords * 16];  // word of the tile << 4 | field
    __shared__ uint16_t s_cc[kTileWords];         // fields that were non-zero at the step's start
    __shared__ uint32_t s_new[kTileWords];        // fields with a non-zero result
    __shared__ uint32_t s_edge[DX ? 1 : kTileWords];  // the same of the word's first and last cell
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gl = lane & (LPW - 1);
    const unsigned group = (0xffffffffu >> (32 - LPW)) << (lane & ~(LPW - 1));
    FaceWriter out(s_buf[warp], nlist, ncount);
    for (int tile = blockIdx.x; tile < S.tiles; tile += gridDim.x) {
        const int bx = box_of_tile(S, tile);
        const BoxDev<T>& B = S.b[bx];
        const Dims& g = B.g;
        const int w0 = (tile - B.tile0) * S.tw, nw = min(S.tw, B.words - w0);
        const int t0 = threadIdx.x;
        uint32_t act = 0, out_old = 0;
        if (t0 < nw) {
            int wlo, whi;
            s_place[t0] = place_word(B, w0 + t0, d, dn, wlo, whi);
            const uint16_t* __restrict__ in = nz_in(B, PH);
            out_old = nz_out(B, PH)[w0 + t0];
            const uint32_t beside = DX ? B.nze[wlo] >> 16 | (B.nze[whi] & 0xffffu) : (uint32_t)in[wlo] | in[whi];
            act = (in[w0 + t0] | beside | out_old) & ((1u << B.K) - 1u);
            if (PH > 0) s_cc[t0] = PH == 2 ? (uint16_t)out_old : B.nzc[w0 + t0];
            s_new[t0] = 0u;
            if (!DX) s_edge[t0] = 0u;
        }
        // the tile's items, word by word
        const int cnt = __popc(act);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        int n = 0, first = incl - cnt;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            if (w < warp) first += s_warp[w];
            n += s_warp[w];
        }
        for (uint32_t m = act; m; m &= m - 1u) s_item[first++] = (uint16_t)(t0 << 4 | (__ffs(m) - 1));
        __syncthreads();
        const T* __restrict__ ud = B.u + (size_t)d * g.N;
        const T* __restrict__ udn = B.u + (size_t)dn * g.N;
        for (int base = warp * WPW; base < n; base += WARPS * WPW) {
            const int idx = base + lane / LPW;
            const bool ok = idx < n;
            const int item = s_item[ok ? idx : base];
            const int t = item >> 4, f = item & 15;
            const WordPlace& p = s_place[t];
            const bool valid = ok && p.i0 + gl * VW < g.nx;
            // lanes past a row's end work on the word's first cell and write nothing
            const int i = p.i0 + (valid ? gl * VW : 0), x = p.x0 + (valid ? gl * VW : 0);
            const int hi = p.hi;
            const bool row_end = i + VW == g.nx;
            const int xn = row_end ? x + VW - g.nx : x + VW;  // the cell after the lane's last along x
            const T* __restrict__ cf = sweep_in(B, PH) + (size_t)f * g.N;
            T cx[VW], cl[VW], ch[VW], ulo[VW], uhi[VW], unl[VW], unh[VW];
            ldv<VW>(cf + x, cx);
            ldv<VW>(ud + x, ulo);
            ldv<VW>(udn + x, unl);
            uint32_t ccw = 0;
            const size_t word = (size_t)f * B.words + w0 + t;
            if (PH > 0 && ok && ((s_cc[t] >> f) & 1u)) ccw = B.ccbits[word];
            if (!DX) {
                ldv<VW>(cf + x + p.lo, cl);
                ldv<VW>(cf + x + hi, ch);
                ldv<VW>(ud + x + hi, uhi);
            }
            if (dn != 0) ldv<VW>(udn + x + p.hin, unh);
            if (DX) {
                const bool need_prev = gl == 0, need_next = gl == LPW - 1 || row_end;
                T cp = __shfl_up_sync(0xffffffffu, cx[VW - 1], 1), cn = __shfl_down_sync(0xffffffffu, cx[0], 1);
                T un = __shfl_down_sync(0xffffffffu, ulo[0], 1);
                if (need_prev) cp = cf[i == 0 ? x + g.nx - 1 : x - 1];
                if (need_next) {
                    cn = cf[xn];
                    un = ud[xn];
                }
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    cl[e] = e == 0 ? cp : cx[e - 1];
                    ch[e] = e == VW - 1 ? cn : cx[e + 1];
                    uhi[e] = e == VW - 1 ? un : ulo[e + 1];
                }
            }
            if (dn == 0) {
                const T un = next_along_x<T, VW>(unl, udn, x, i, g.nx, gl, LPW);
#pragma unroll
                for (int e = 0; e < VW; ++e) unh[e] = e == VW - 1 ? un : unl[e + 1];
            }
            uint32_t ccm = 0;
            if (PH == 0) {
                if (valid) {
#pragma unroll
                    for (int e = 0; e < VW; ++e) ccm |= (above_half(cx[e]) ? 1u : 0u) << e;
                }
                const uint32_t w = gather_word<VW>(ccm, lane);
                if (ok && gl == 0) B.ccbits[word] = w;
            } else {
                ccm = (ccw >> ((gl * VW) & 31)) & ((1u << VW) - 1u);
            }
            T v[VW], rem[VW];
            uint32_t flo = 0, fhi = 0, occm = 0;
            bool nonzero = false, clipped = false;
            const T* __restrict__ flux = B.flux + (size_t)f * g.N;
            // upwind donors through the low and high faces: empty (no flux),
            // full (flux s) or interfacial (the listed flux)
            bool change[VW], full_lo[VW], full_hi[VW];
            T F_lo[VW], F_hi[VW];
            bool any = false;
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                const int sl = vsign(ulo[e]), sh = vsign(uhi[e]);
                const T dl = sl > 0 ? cl[e] : cx[e], dh = sh < 0 ? ch[e] : cx[e];
                const bool ml = valid && sl != 0 && holds<VW>(dl), mh = valid && sh != 0 && holds<VW>(dh);
                full_lo[e] = ml && at_least_one(dl);
                full_hi[e] = mh && at_least_one(dh);
                F_lo[e] = F_hi[e] = T(0);
                if (ml && !full_lo[e]) F_lo[e] = flux[x + e];
                if (mh && !full_hi[e]) F_hi[e] = flux[DX ? (e < VW - 1 ? x + e + 1 : xn) : x + e + hi];
                change[e] = ml || mh || ((ccm >> e) & 1u);
                any = any || change[e];
                v[e] = cx[e];
            }
            // the arithmetic once for the warp, its cases by selects (branches
            // ran it with four lanes at a time: in double the FP64 pipe was
            // 79% busy at a tenth of its lanes)
            if (__any_sync(0xffffffffu, any)) {
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    const T s_lo = mul_rn(ulo[e], B.sfac), s_hi = mul_rn(uhi[e], B.sfac);
                    const T lo = full_lo[e] ? s_lo : F_lo[e], hi_ = full_hi[e] ? s_hi : F_hi[e];
                    const T r = cx[e] - (hi_ - lo), rc = r + (s_hi - s_lo);
                    if (change[e]) v[e] = (ccm >> e) & 1u ? rc : r;
                }
            }
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                rem[e] = T(0);
                if (PH == 2) {
                    const bool under = below_zero(v[e]), over = above(v[e], T(1));
                    if ((under || over) && valid) {
                        // v - 0 and v - 1 are exact (Sterbenz): the FP64 sum
                        // below has the terms of FP64 differences
                        const T end = under ? T(0) : T(1);
                        rem[e] = v[e] - end;
                        v[e] = end;
                        clipped = true;
                    }
                    occm |= (valid && above(v[e], tau) ? 1u : 0u) << e;
                }
                nonzero |= !is_exact_zero(v[e]);
                if (holds<VW>(v[e]) && !at_least_one(v[e])) {
                    flo |= (valid && vsign(unl[e]) < 0 ? 1u : 0u) << e;
                    fhi |= (valid && vsign(unh[e]) > 0 ? 1u : 0u) << e;
                }
            }
            if (valid) stv<VW>(sweep_out(B, PH) + (size_t)f * g.N + x, v);
            const unsigned vote = __ballot_sync(0xffffffffu, valid && nonzero);
            if (ok && gl == 0 && (vote & group)) atomicOr(&s_new[t], 1u << f);
            if (!DX && dn == 0 && valid) {
                if (gl == 0 && !is_exact_zero(v[0])) atomicOr(&s_edge[t], 1u << f);
                if (i + VW == min(p.i0 + 32, g.nx) && !is_exact_zero(v[VW - 1])) atomicOr(&s_edge[t], 0x10000u << f);
            }
            if (PH == 2) {
                const uint32_t w = gather_word<VW>(occm, lane);
                if (ok && gl == 0) B.occbits[word] = w;
                if (__any_sync(0xffffffffu, clipped)) {
                    double removed = 0.0;
#pragma unroll
                    for (int e = 0; e < VW; ++e) removed += (double)rem[e];
#pragma unroll
                    for (int o = LPW / 2; o > 0; o >>= 1) removed += __shfl_down_sync(0xffffffffu, removed, o, LPW);
                    if (ok && gl == 0 && !is_exact_zero(removed)) atomicAdd(B.clipped + f, removed);
                }
            }
            const int nflag = __popc(flo) + __popc(fhi);
            if (__any_sync(0xffffffffu, nflag != 0)) {
                int pos = out.reserve(nflag, lane);
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    if ((flo >> e) & 1u) out.buf[pos++] = face_key(bx, f, 0, x + e);
                    if ((fhi >> e) & 1u) out.buf[pos++] = face_key(bx, f, 1, x + e);
                }
                out.settle(lane);
            }
        }
        __syncthreads();
        // the output's map; fields past K keep their bits
        if (t0 < nw) {
            const uint32_t m = s_new[t0] | (out_old & ~((1u << B.K) - 1u));
            if (m != out_old) nz_out(B, PH)[w0 + t0] = (uint16_t)m;
            if (!DX && dn == 0) B.nze[w0 + t0] = s_edge[t0];
        }
        // (the next tile's first barrier comes before anything reads what its
        // build writes, and this thread's s_new and s_edge are read above by itself)
    }
    out.flush(lane);
}

template <typename T, int NB, int VW>
static void launch_update_vw(const BoxSet<T, NB>& S, int d, int dn, int sweep, T tau, unsigned long long* nlist,
                             int* ncount, int gb, cudaStream_t st) {
    auto go = [&](auto kernel) { kernel<<<gb, kSweepThreads, 0, st>>>(S, d, dn, tau, nlist, ncount); };
    if (sweep == 0) d == 0 ? go(k_update_sp<T, NB, VW, 0, true>) : go(k_update_sp<T, NB, VW, 0, false>);
    else if (sweep == 1) d == 0 ? go(k_update_sp<T, NB, VW, 1, true>) : go(k_update_sp<T, NB, VW, 1, false>);
    else d == 0 ? go(k_update_sp<T, NB, VW, 2, true>) : go(k_update_sp<T, NB, VW, 2, false>);
}

// Launch of the update pass of sweep `sweep` (0, 1, 2) along d; vec: VecOf<T>
// cells per lane (whole 16-byte lanes), else one.
template <typename T, int NB>
static cudaError_t launch_update(const BoxSet<T, NB>& S, bool vec, int d, int dn, int sweep, T tau,
                                 unsigned long long* nlist, int* ncount, int gb, cudaStream_t st) {
    if (vec) {
        launch_update_vw<T, NB, VecOf<T>::W>(S, d, dn, sweep, tau, nlist, ncount, gb, st);
    } else {
        if constexpr (NB == 1) launch_update_vw<T, NB, 1>(S, d, dn, sweep, tau, nlist, ncount, gb, st);
    }
    return cudaGetLastError();
}
template <typename T, int NB>
static void launch_list(const BoxSet<T, NB>& S, bool vec, int d, T tau, unsigned long long* list, int* count, int gb,
                        cudaStream_t st) {
    if (vec) {
        k_list_sp<T, NB, VecOf<T>::W><<<gb, kSweepThreads, 0, st>>>(S, d, tau, list, count);
    } else {
        if constexpr (NB == 1) k_list_sp<T, NB, 1><<<gb, kSweepThreads, 0, st>>>(S, d, tau, list, count);
    }
}

// Resident blocks per SM of the y/z update pass, queried on the kernel copy
// of the unit that launches it (no relocatable device code).
template <typename T, int NB, int VW>
static int update_blocks_per_sm() {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_update_sp<T, NB, VW, 1, false>, kSweepThreads, 0) !=
        cudaSuccess)
        per_sm = 0;
    (void)cudaGetLastError();
    return per_sm;
}

// A listed face of a box set: box, field, upwind donor, the cell x of the
// face's high side and the flux index t = f N + x.
struct BoxFace {
    int box, f, x, donor;
    int di, dj, dk;  // the donor's cell coordinates
    size_t t;
};

template <typename T, int NB>
__device__ __forceinline__ BoxFace decode_box_face(const BoxSet<T, NB>& S, unsigned long long key, int d) {
    BoxFace r;
    r.box = NB == 1 ? 0 : (int)(key >> 36);
    r.f = (int)((key >> kFaceFieldShift) & 15u);
    const BoxDev<T>& B = S.b[r.box];
    const Dims& g = B.g;
    r.donor = (int)((uint32_t)key & 0x7fffffffu);
    const int row = (int)fastdiv((uint32_t)r.donor, B.divnx);
    r.di = r.donor - row * g.nx;
    r.dk = (int)fastdiv((uint32_t)row, B.divny);
    r.dj = row - r.dk * g.ny;
    r.x = r.donor;
    if ((uint32_t)key >> 31) r.x = step_cell(r.donor, r.di, r.dj, r.dk, d, 1, g);
    r.t = (size_t)r.f * g.N + r.x;
    return r;
}
// The face's velocity along d.
template <typename T, int NB>
__device__ __forceinline__ T face_velocity(const BoxSet<T, NB>& S, const BoxFace& fc, int d) {
    const BoxDev<T>& B = S.b[fc.box];
    return B.u[(size_t)d * B.g.N + fc.x];
}

// After Step 4 moved drops (one box): every face of the current list (the
// next sweep's faces, direction d, whose upwind donor is interfacial) whose
// donor is a cell of a moving drop now belongs to the drop's target field.
// A moved cell keeps its value and only changes field, and the target
// field held nothing occupied within reach of the drop, so the rest of the
// list stands (a target cell that held a residue below the occupancy
// threshold may end up listed twice, which writes the same flux twice).  A
// donor's tag is read only where the Step 1 snapshot marks it occupied.
template <typename T>
__global__ void __launch_bounds__(256) k_list_patch(const __grid_constant__ BoxSet<T, 1> S, int d,
                                                    unsigned long long* __restrict__ list,
                                                    const int* __restrict__ count,
                                                    const uint32_t* __restrict__ bits,
                                                    const int* __restrict__ labels, MoveTables mt,
                                                    const int* __restrict__ target) {
    const Dims& g = S.b[0].g;
    const size_t wpf = (size_t)g.rows * g.W;
    const int n = *count;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const unsigned long long key = list[e];
        const int f = (int)((key >> kFaceFieldShift) & 15u);
        if (mt.mv_count[f] == 0) continue;
        const BoxFace fc = decode_box_face(S, key, d);
        const size_t row = (size_t)fc.dk * g.ny + fc.dj;
        if (!((bits[(size_t)f * wpf + row * g.W + (fc.di >> 5)] >> (fc.di & 31)) & 1u)) continue;
        const int l = labels[(size_t)f * g.N + fc.donor];
        if (!is_moving(mt, f, l)) continue;
        const int m = moving_index(mt, f, l);
        const int tg = m >= 0 ? target[m] : -1;
        if (tg >= 0) list[e] = (key & ~(15ull << kFaceFieldShift)) | ((unsigned long long)tg << kFaceFieldShift);
    }
}

// MYC fluxes of the listed faces of every box (one thread per face);
// *next_count, the count of the list that the sweep's update pass will fill, is
// set to zero.
//
// In double the kernel is bound by FP64 issue (1/64 of the FP32 rate), so
// its time is its count of FP64 warp instructions: the forms of plic64.cuh, and
// the roots taken by piece (cubic, square root, cube root: the block's faces are
// reordered so that a warp runs one piece, at most two, instead of all three
// with nine lanes each), took it from 6.2 to 0.72 ms per sweep of the 256^3,
// K = 8, phi = 0.3 box (2.7 M faces; 1.08 ms before the reordering and before
// the volume's pieces became selects), and a sweep of 32^3 with 8 drops, where
// one warp's chain is the time, from 78 to 20 us with its other launches.  0.55 ms
// since the normals near a tie go to a call and fluxes of donors a few ulps from
// 1 do without (84 FP64 instructions per warp of faces in the first sweep).
//
// In FP32 the faces whose fraction lies within `band` of 0 or 1 (one in six)
// take an FP64 step: they are compacted to the first threads of the block, so
// that one warp in four issues it (the FP64 pipe was 57 to 69% busy with every
// warp doing so: 66 -> 56 us per sweep at 192 x 160 x 224, K = 6).
template <typename T, int NB>
__global__ void __launch_bounds__(kFaceTile) k_face_flux_bx(const __grid_constant__ BoxSet<T, NB> S, int d,
                                                            int sweep, T band,
                                                            const unsigned long long* __restrict__ list,
                                                            const int* __restrict__ count,
                                                            int* __restrict__ next_count) {
    constexpr bool kBanded = std::is_same<T, float>::value;
    constexpr int kWarps = kFaceTile / 32;
    __shared__ T s_q[4][kFaceTile];  // queued normals and fractions (a piece's variables), then constants
    __shared__ int s_n[kWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (blockIdx.x == 0 && t == 0) *next_count = 0;
    const int n = *count;
    for (int base = blockIdx.x * kFaceTile; base < n; base += gridDim.x * kFaceTile) {
        const bool valid = base + t < n;
        T m[3] = {T(1), T(0), T(0)}, cv = T(0.5), sv = T(0);
        T* dst = nullptr;
        if (valid) {
            const BoxFace fc = decode_box_face(S, list[base + t], d);
            const BoxDev<T>& B = S.b[fc.box];
            sv = face_velocity(S, fc, d) * B.sfac;
            dst = B.flux + fc.t;
            T st[27];
            gather_stencil_ijk(sweep_in(B, sweep) + (size_t)fc.f * B.g.N, fc.di, fc.dj, fc.dk, B.g, st);
            cv = st[13];
            if constexpr (kBanded) myc_normal(st, m);
            else myc_direction64(st, m, kFluxEdge);
        }
        if constexpr (kBanded) {
            const bool queue = valid && (cv < band || cv > T(1) - band);
            const unsigned vote = __ballot_sync(0xffffffffu, queue);
            if (lane == 0) s_n[warp] = __popc(vote);
            __syncthreads();
            int at = __popc(vote & ((1u << lane) - 1u)), nq = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                at += w < warp ? s_n[w] : 0;
                nq += s_n[w];
            }
            if (queue) {
                s_q[0][at] = m[0];
                s_q[1][at] = m[1];
                s_q[2][at] = m[2];
                s_q[3][at] = cv;
            }
            __syncthreads();
            if (t < nq) s_q[3][t] = plic_alpha_banded(s_q[0][t], s_q[1][t], s_q[2][t], s_q[3][t], band);
            T alpha = T(0);
            if (valid && !queue) alpha = plic_alpha<T>(m[0], m[1], m[2], cv);
            __syncthreads();
            if (queue) alpha = s_q[3][at];
            if (valid) *dst = face_flux(m, alpha, d, sv);
            // (s_q is written again only after the next tile's first barrier)
        } else {
            // the roots by piece: the faces of a piece on neighbouring threads
            T a = abs64(m[0]), b = abs64(m[1]), c = abs64(m[2]);
            sort3_pos(a, b, c);
            const bool flip = lt_pos(T(0.5), cv);
            T p, w6, g, x;
            const int piece = valid ? alpha64_piece(a, b, c, flip ? T(1) - cv : cv, p, w6, g, x) : kAlphaLinear;
            const unsigned v0 = __ballot_sync(0xffffffffu, piece == 0), v1 = __ballot_sync(0xffffffffu, piece == 1),
                           v2 = __ballot_sync(0xffffffffu, piece == 2);
            if (lane == 0) s_n[warp] = __popc(v0) | __popc(v1) << 8 | __popc(v2) << 16;
            __syncthreads();
            int before = 0, all = 0;  // three counts of up to 128, 8 bits each
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                before += w < warp ? s_n[w] : 0;
                all += s_n[w];
            }
            const int n0 = all & 255, n1 = n0 + (all >> 8 & 255), n2 = n1 + (all >> 16);
            const unsigned mine = piece == 0 ? v0 : (piece == 1 ? v1 : v2);
            const int at = (piece == 0 ? 0 : (piece == 1 ? n0 : n1)) + (before >> (8 * piece) & 255) +
                           __popc(mine & ((1u << lane) - 1u));
            if (piece != kAlphaLinear) {
                s_q[0][at] = p;
                s_q[1][at] = w6;
                s_q[2][at] = g;
            }
            __syncthreads();
            if (t < n2) s_q[3][t] = alpha64_root(t < n0 ? 0 : (t < n1 ? 1 : 2), s_q[0][t], s_q[1][t], s_q[2][t]);
            __syncthreads();
            if (piece != kAlphaLinear) x = b * s_q[3][at];
            if (valid) *dst = face_flux64_at(m, flip ? (a + b + c) - x : x, d, sv);
        }
    }
}

}  // namespace vof
