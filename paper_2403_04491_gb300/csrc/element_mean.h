// Mean of an element's D + 1 vertex values from their sum (host and device).
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define KNP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define KNP_HOST_DEVICE inline
#endif

namespace knp {

// s / (D + 1), D + 1 = 3 or 4, without an FP64 division (some 20 instructions of the slow pipe each: 833 us
// of k_elem_means at 128^3, now 365 us): a quarter is exact; a third is the product with the rounded third and one
// FMA of its remainder, Markstein's correction, which gives the correctly rounded quotient of a finite s. The
// remainder of an infinite s or a NaN is a NaN, that of a zero a zero of either sign: those keep the product.
template <int D>
KNP_HOST_DEVICE double mean_of_sum(double s) {
    if (D == 3) return 0.25 * s;
    const double third = 1.0 / 3.0, q = s * third;
    const double r = fma(-3.0, q, s);
    return fabs(r) > 0.0 ? fma(r, third, q) : q;
}

}  // namespace knp
