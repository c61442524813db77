// Row products by groups of lanes: how many lanes work on a row, and how their sums are combined.
#pragma once

#include <cstdint>

namespace knp {

// Lanes per row of a row-product kernel over a sliced-ELL pattern: 1, 4 or 8. One thread per row
// suffices once the rows alone give every SM enough loads in flight; a smaller matrix leaves the
// SMs waiting on each row's chain of dependent loads, which 4 or 8 lanes shorten by that factor.
// Lanes are added while the grid stays below LANE_THREADS (the threads that give 152 SMs 16 warps
// each) and every lane keeps at least one entry of a mean row. Chebyshev step of the FP64 hierarchy,
// one lane against several: 1,153 rows of 7 entries 9.3 -> 5.2 us (8 lanes), 29,376 rows of 14
// entries 17.5 -> 10.8 us (4 lanes).
constexpr int64_t LANE_THREADS = 152 * 512;
inline int row_lanes(int64_t rows, double mean_len) {
    if (rows >= LANE_THREADS) return 1;
    return (8 * rows <= LANE_THREADS && mean_len > 4.0) ? 8 : 4;
}

// Sums of the four fields over the L lanes of a row (consecutive lanes of one warp, L a power of
// two): on return out[0 .. LANE_FIELDS<L>) are the fields from lane_field<L>(t) on; the lanes from 4 on
// hold copies. A reduce-scatter: each halving step exchanges half of the values, so 4 lanes take
// 3 shuffles and 3 adds instead of 8 (the adds of doubles are the scarce ones).
template <int L>
constexpr int LANE_FIELDS = L >= 4 ? 1 : 4 / L;
template <int L>
__device__ __forceinline__ int lane_field(int t) {
    return L == 1 ? 0 : L == 2 ? 2 * t : (t & 3);
}
template <class T, int L>
__device__ __forceinline__ void lane_reduce4(const T acc[4], int t, T* out) {
    if constexpr (L == 1) {
#pragma unroll
        for (int f = 0; f < 4; ++f) out[f] = acc[f];
    } else {
        constexpr int O = L == 2 ? 1 : 2;
        const bool hi = (t & O) != 0;
        T a0 = hi ? acc[2] : acc[0], a1 = hi ? acc[3] : acc[1];
        const T b0 = hi ? acc[0] : acc[2], b1 = hi ? acc[1] : acc[3];
        a0 += __shfl_xor_sync(0xffffffffu, b0, O);
        a1 += __shfl_xor_sync(0xffffffffu, b1, O);
        if constexpr (L == 2) {
            out[0] = a0;
            out[1] = a1;
        } else {
            const bool odd = (t & 1) != 0;
            T a = odd ? a1 : a0;
            a += __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 1);
#pragma unroll
            for (int o = 4; o < L; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            out[0] = a;
        }
    }
}

}  // namespace knp
