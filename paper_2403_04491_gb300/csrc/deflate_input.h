// The coarse correction's input at one node, shared by its own pass and the V-cycle's first kernel.
#pragma once

#include "vcycle.h"

namespace knp {

// t = s .* v - (A Z y)_i, or - (A^T Z y)_i. Only an active row (df.act) has a nonzero A Z y: its fixed
// coefficients times its own group's constant and the one on the membrane's other side. (Forming it from
// the row's cross-region entries here made every warp that meets an active row pay for the longest of
// its entry loops: 126 us at 128^3, 104 us of it FP64 issue; now 82 us.)
__device__ __forceinline__ void defl_input(int64_t i, const double* __restrict__ v, const double* __restrict__ s,
                                           const DeflFuse& df, double t[4]) {
    const double2* vp = reinterpret_cast<const double2*>(v + 4 * i);
    const double2* sp = reinterpret_cast<const double2*>(s + 4 * i);
    const int32_t a = df.act[i];
    const double2 v0 = vp[0], v1 = vp[1], s0 = sp[0], s1 = sp[1];
    t[0] = s0.x * v0.x;
    t[1] = s0.y * v0.y;
    t[2] = s1.x * v1.x;
    t[3] = s1.y * v1.y;
    if (a < 0) return;
    const double yo = df.y[i < df.N_i ? df.rgrp[i] : df.ext_group], yc = df.y[df.xgrp[a]];
    const double* c = df.C + 8 * (int64_t)a;
    for (int q = 0; q < 4; ++q) t[q] -= c[q] * yo + c[4 + q] * yc;
}

}  // namespace knp
