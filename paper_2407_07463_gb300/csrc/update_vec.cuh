// Lane helpers of the sweep passes: a lane owns VW consecutive cells of a row
// (4 floats or 2 doubles, one 16-byte access, or a single cell where rows are
// not whole 16-byte lanes), a group of 32 / VW lanes a word of 32 cells.
// Neighbours along x come from the adjacent lane by a shuffle (or from memory
// at the group's ends and the periodic boundary); c_c and occupancy bit words
// are assembled with shuffles.
#pragma once

#include "common.cuh"

namespace vof {

template <typename T>
struct VecOf;
template <>
struct VecOf<float> {
    static constexpr int W = 4;
};
template <>
struct VecOf<double> {
    static constexpr int W = 2;
};

template <typename T>
__device__ __forceinline__ void ld16(const T* __restrict__ p, T v[16 / sizeof(T)]) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else {
        const double2 q = __ldg(reinterpret_cast<const double2*>(p));
        v[0] = q.x;
        v[1] = q.y;
    }
}

template <typename T>
__device__ __forceinline__ void st16(T* p, const T v[16 / sizeof(T)]) {
    if constexpr (sizeof(T) == 4)
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}

// VW consecutive values: one 16-byte access, or one value.
template <int VW, typename T>
__device__ __forceinline__ void ldv(const T* __restrict__ p, T v[VW]) {
    if constexpr (VW == 1) v[0] = __ldg(p);
    else ld16(p, v);
}
template <int VW, typename T>
__device__ __forceinline__ void stv(T* p, const T v[VW]) {
    if constexpr (VW == 1) *p = v[0];
    else st16(p, v);
}

// Value of the cell after the lane's last one along x (periodic in the row);
// gl: the lane's place in its group of lpw lanes.
template <typename T, int VW>
__device__ __forceinline__ T next_along_x(const T v[VW], const T* __restrict__ arr, int x, int i, int nx, int gl,
                                          int lpw) {
    T n = __shfl_down_sync(0xffffffffu, v[0], 1);
    const bool row_end = i + VW == nx;
    if (gl == lpw - 1 || row_end) n = arr[row_end ? x + VW - nx : x + VW];
    return n;
}

// OR of the lanes' VW-bit masks into 32-bit words: lane 0 of each group of
// 32 / VW lanes returns the word of its group.
template <int VW>
__device__ __forceinline__ uint32_t gather_word(uint32_t bits, int lane) {
    uint32_t w = bits << ((lane * VW) & 31);
#pragma unroll
    for (int o = 1; o < 32 / VW; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
    return w;
}

}  // namespace vof
