// Listed-face helpers shared by the sweep kernels (internal).
#pragma once

#include "common.cuh"

namespace vof {

// 3x3x3 stencil of cell (i, j, k) (periodic), st[(k+1)*9 + (j+1)*3 + (i+1)].
template <typename T>
__device__ __forceinline__ void gather_stencil_ijk(const T* __restrict__ cf, int i, int j, int k, const Dims& g,
                                                   T st[27]) {
    int im = i == 0 ? g.nx - 1 : i - 1, ip = i == g.nx - 1 ? 0 : i + 1;
    int jm = j == 0 ? g.ny - 1 : j - 1, jp = j == g.ny - 1 ? 0 : j + 1;
    int km = k == 0 ? g.nz - 1 : k - 1, kp = k == g.nz - 1 ? 0 : k + 1;
    const int is[3] = {im, i, ip}, js[3] = {jm, j, jp}, ks[3] = {km, k, kp};
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int a = 0; a < 3; ++a) st[c * 9 + b * 3 + a] = cf[cell(is[a], js[b], ks[c], g)];
}

// A warp's way into a face list: entries gather in the warp's own shared
// buffer and go to the list in runs of more than kWarpFill, with one
// atomicAdd on the list's count and coalesced stores, so that the list has no
// gaps and a consumer's entry e is list[e].  (Segments per block, found by an
// offset scan, a launch of its own, and a lookup per tile, cost 5 to 30 us
// per sweep.)  An append adds at most 256 entries (4 words of 32 cells with 2
// faces each).
constexpr int kWarpFill = 128, kWarpBuf = kWarpFill + 256;
struct FaceWriter {
    unsigned long long* buf;   // [kWarpBuf] in shared memory
    unsigned long long* list;
    int* count;                // entries of the list
    int n = 0;                 // entries in buf, the same on every lane
    __device__ __forceinline__ FaceWriter(unsigned long long* b, unsigned long long* l, int* c)
        : buf(b), list(l), count(c) {}
    // Place for `own` entries of this lane in buf; every lane calls it.
    __device__ __forceinline__ int reserve(int own, int lane) {
        int incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int at = n + incl - own;
        n += __shfl_sync(0xffffffffu, incl, 31);
        return at;
    }
    // After the reserved entries are written (every lane): makes room.
    __device__ __forceinline__ void settle(int lane) {
        if (n > kWarpFill) flush(lane);
    }
    __device__ __forceinline__ void flush(int lane) {
        if (n == 0) return;
        __syncwarp();
        int base = 0;
        if (lane == 0) base = atomicAdd(count, n);
        base = __shfl_sync(0xffffffffu, base, 0);
        for (int q = lane; q < n; q += 32) list[(size_t)base + q] = buf[q];
        n = 0;
        __syncwarp();
    }
};

}  // namespace vof
