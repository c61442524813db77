// The coarse correction's input at one node, shared by its own pass and the V-cycle's first kernel.
#pragma once

#include "vcycle.h"

namespace knp {

// t = s .* v - (A Z y)_i, or - (A^T Z y)_i. Only an active row (df.act) has a nonzero A Z y: its
// same-region phi columns hold its own group's constant (the row sums RS), its cross-region entries
// their groups' constants; the potential row is sum_k z_k of the concentration rows' terms. In the
// transposed operator the concentration rows see tau_r^k z_k times the row sum of a, and the potential
// row sum_k z_k e^k, with the cross entries in the transposed list. The pinned potential row (the
// identity) gives 0.
__device__ __forceinline__ void defl_input(int64_t i, const double* __restrict__ v, const double* __restrict__ s,
                                           const DeflFuse& df, double t[4]) {
    const double2* vp = reinterpret_cast<const double2*>(v + 4 * i);
    const double2* sp = reinterpret_cast<const double2*>(s + 4 * i);
    const double2 v0 = vp[0], v1 = vp[1], s0 = sp[0], s1 = sp[1];
    t[0] = s0.x * v0.x;
    t[1] = s0.y * v0.y;
    t[2] = s1.x * v1.x;
    t[3] = s1.y * v1.y;
    const int32_t a = df.act[i];
    if (a < 0) return;
    const bool in = i < df.N_i;
    const double yr = df.y[in ? df.rgrp[i] : df.ext_group];
    double ae[3];
    for (int q = 0; q < 3; ++q) ae[q] = df.RS[3 * (int64_t)a + q] * yr;
    for (int u = df.xptr[i]; u < df.xptr[i + 1]; ++u) {
        const int gq = df.xg[u];
        if (gq < 0) continue;
        const int64_t idx = df.transpose ? df.xidx[u] : u;
        const double yc = df.y[gq];
        for (int q = 0; q < 3; ++q) ae[q] += df.xe[q * df.n_cross + idx] * yc;
    }
    if (i != df.pin) t[3] -= df.z[0] * ae[0] + df.z[1] * ae[1] + df.z[2] * ae[2];
    if (df.transpose) {
        const double ay = df.RSa[a] * yr;
        for (int q = 0; q < 3; ++q) t[q] -= df.ztau[in ? 0 : 1][q] * ay;
    } else {
        for (int q = 0; q < 3; ++q) t[q] -= ae[q];
    }
}

}  // namespace knp
