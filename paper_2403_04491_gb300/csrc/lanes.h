// Row products by groups of lanes: how many lanes work on a row, and how their sums are combined.
#pragma once

#include <cstdint>

namespace knp {

// Lanes per row of a row-product kernel over a sliced-ELL pattern: 1, 4 or 8. More lanes shorten a row's
// chain of dependent loads, which is what a small matrix waits for; but each row's sums over the lanes, its
// epilogue and lanes without an entry are FP64 instructions that one thread per row does not issue. One
// thread per row is better once the rows are many for their length, 18 per SM and entry (2D, 7 entries: from
// 19,200 rows, 3D, 14.5: from 39,700), and always from LANE_THREADS on, where the rows alone fill the SMs.
// Three time steps (rtol 1e-11) with four lanes and with one, by the finest level's rows per SM and entry:
//     2D  12.0  5.10  5.32 ms    15.2  6.20  6.10    18.7  6.95  6.55    22.0  8.81  7.86    31.5  11.3  10.1
//     3D  10.7  7.08  7.32       14.4  8.91  8.83    17.2  9.40  9.40    20.5  11.3  11.1    32.5  14.7  13.3
// (the 2D pass at 22.0 also in four iterations less of 86); at 15 P2 on 80x80 (27,000 rows of 11.5) is 5% slower
// with one. Eight lanes up to 4,864 rows; three steps by the finest level's rows:
//     2D   1,153  eight 2.10, four 2.12 ms     3,841  4.30, 4.27     5,473  4.25, 4.05     7,568  4.41, 4.01
//     3D   1,429  eight 2.43, four 2.49        4,314  2.86, 2.78     6,128  4.40, 4.19     8,296  5.16, 4.69
// Below the limit the two are within 3% of each other and neither always ahead: the Kir problem on 97x75 is 3%
// slower with four (its first coarse level).
constexpr int64_t LANE_THREADS = 152 * 512;
inline int row_lanes(int64_t rows, double mean_len) {
    if (rows >= LANE_THREADS || rows >= 152 * 18 * mean_len) return 1;
    return (16 * rows <= LANE_THREADS && mean_len > 4.0) ? 8 : 4;
}

// Sums of the four fields over the L lanes of a row (consecutive lanes of one warp, L = 1 or a power of
// two from 4): on return out[0 .. LANE_FIELDS<L>) are the fields from lane_field<L>(t) on; the lanes from 4 on
// hold copies. A reduce-scatter: each halving step exchanges half of the values, so 4 lanes take
// 3 shuffles and 3 adds instead of 8 (the adds of doubles are the scarce ones).
template <int L>
constexpr int LANE_FIELDS = L >= 4 ? 1 : 4;
template <int L>
__device__ __forceinline__ int lane_field(int t) {
    return L == 1 ? 0 : (t & 3);
}
template <class T, int L>
__device__ __forceinline__ void lane_reduce4(const T acc[4], int t, T* out) {
    static_assert(L == 1 || L >= 4, "lanes per row");
    if constexpr (L == 1) {
#pragma unroll
        for (int f = 0; f < 4; ++f) out[f] = acc[f];
    } else {
        const bool hi = (t & 2) != 0, odd = (t & 1) != 0;
        T a0 = hi ? acc[2] : acc[0], a1 = hi ? acc[3] : acc[1];
        const T b0 = hi ? acc[0] : acc[2], b1 = hi ? acc[1] : acc[3];
        a0 += __shfl_xor_sync(0xffffffffu, b0, 2);
        a1 += __shfl_xor_sync(0xffffffffu, b1, 2);
        T a = odd ? a1 : a0;
        a += __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 1);
#pragma unroll
        for (int o = 4; o < L; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        out[0] = a;
    }
}

}  // namespace knp
