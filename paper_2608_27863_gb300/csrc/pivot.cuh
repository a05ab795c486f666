// Pivot step shared by the elimination kernels: the search by one warp and the
// reciprocal by one lane.  An FP64 instruction of a warp holds its SM's pipe for
// 16 cycles and queues behind the trailing updates of the other warps, so
// magnitudes are compared as integers and the division is done once, not by
// every thread (512 hexes p = 2, FP64 elimination before the Schur product: 7.22 -> 6.9 ms;
// 64 quads p = 2, 128 -> 107 us).
#pragma once

#include <climits>

namespace hdg {

// order of |v| as an integer: larger magnitude, larger key; NaN 0, everything else at least 1
__device__ __forceinline__ unsigned long long pivot_key(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
    return u > 0x7FF0000000000000ull ? 0ull : u + 1ull;
}
__device__ __forceinline__ unsigned pivot_key(float v) {
    const unsigned u = __float_as_uint(v) & 0x7FFFFFFFu;
    return u > 0x7F800000u ? 0u : u + 1u;
}

// row in [r0, r1) of largest |val(row)|, the lowest row on ties; INT_MAX when every value is NaN.
// One whole warp; the result in every lane.
template <class Val>
__device__ __forceinline__ int warp_pivot(int r0, int r1, Val val) {
    const int lane = threadIdx.x & 31;
    decltype(pivot_key(val(0))) bk = 0;
    int bi = INT_MAX;
#pragma unroll 1
    for (int r = r0 + lane; r < r1; r += 32) {
        const auto k = pivot_key(val(r));
        if (k > bk) { bk = k; bi = r; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const auto ok = __shfl_down_sync(0xffffffffu, bk, off);
        const int oi = __shfl_down_sync(0xffffffffu, bi, off);
        if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
    }
    return __shfl_sync(0xffffffffu, bi, 0);
}

// reciprocal of the pivot; a zero or non-finite one counts as one and sets flag 1 or 2 (one thread)
template <class T>
__device__ __forceinline__ T pivot_reciprocal(T pv, int& flag) {
    const auto k = pivot_key(pv);
    constexpr bool F64 = sizeof(T) == 8;
    const bool inf = F64 ? (unsigned long long)k == 0x7FF0000000000001ull : (unsigned)k == 0x7F800001u;
    if (k == 1 || k == 0 || inf) {                      // zero, NaN, infinity
        flag |= k == 1 ? 1 : 2;
        return T(1);
    }
    return T(1) / pv;
}

}  // namespace hdg
