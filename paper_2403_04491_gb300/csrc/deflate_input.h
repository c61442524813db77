// Parts of the coarse correction that other kernels share: the gather's partial sums (its own kernel and the
// orthogonalisation's last), the small solve and the corrected input (their own kernels and the V-cycle's
// first).
#pragma once

#include "vcycle.h"

namespace knp {

constexpr int DT = 256;   // threads of the blocks that call block_sum, gather_share or coarse_solve

// sum over a block of DT threads, valid in thread 0; sh: [DT / 32]
__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < DT / 32; ++w) s += sh[w];
    return s;
}

// Partial sums of g = Z^T r, one per block: blocks [0, nchunks) take one chunk of a cell's nodes each,
// the next ones shares of the extracellular potentials (pin left out)
struct GatherArgs {
    int32_t nchunks = 0, next = 0;
    const int64_t* cbeg = nullptr;     // chunk -> its first entry of cnodes
    const int32_t* cnodes = nullptr;   // intracellular nodes by group
    int64_t N_i = 0, n = 0;
    int32_t pin = -1;
    double* part = nullptr;
};

// This thread's part of block b's sum; value(k): r at position k of the node-major vectors
template <class Value>
__device__ __forceinline__ double gather_share(const GatherArgs& a, int b, Value&& value) {
    double acc = 0.0;
    if (b < a.nchunks) {
        const int64_t end = a.cbeg[b + 1];
        for (int64_t q = a.cbeg[b] + threadIdx.x; q < end; q += DT) acc += value(4 * (int64_t)a.cnodes[q] + 3);
    } else {
        const int64_t stride = (int64_t)a.next * DT;
        for (int64_t r = a.N_i + (b - a.nchunks) * (int64_t)DT + threadIdx.x; r < a.n; r += stride)
            if (r != a.pin) acc += value(4 * r + 3);
    }
    return acc;
}

// y = E^{-1} g by one block of DT threads: y_e = (g_e - sum_j E_ej g_j / E_jj) / S_e,
// y_j = (g_j - E_je y_e) / E_jj; y[nc] = y_e. The division by E_jj and S_e is a product with their
// reciprocals, formed once per step (an FP64 division is a chain of some 20 instructions). y may be shared
// memory; its values are there for the whole block on return.
__device__ __forceinline__ void coarse_solve(const CoarseSolve& e, double* y) {
    __shared__ double sh[DT / 32];
    __shared__ double ye_s;
    double a = 0.0;
    for (int q = threadIdx.x; q < e.next; q += DT) a += e.part[e.nchunks + q];
    // a thread per cell, or a warp where cells have many chunks: g_j (kept in y until the solve)
    const bool wide = e.nchunks > 8 * e.nc;
    const int lane = threadIdx.x & 31;
    for (int j = wide ? threadIdx.x >> 5 : threadIdx.x; j < e.nc; j += wide ? DT / 32 : DT) {
        double g = 0.0;
        for (int q = e.cchunk[j] + (wide ? lane : 0); q < e.cchunk[j + 1]; q += wide ? 32 : 1) g += e.part[q];
        if (wide)
            for (int o = 16; o > 0; o >>= 1) g += __shfl_down_sync(0xffffffffu, g, o);
        if (!wide || lane == 0) {
            y[j] = g;
            a -= e.Eej[j] * (g * e.iEjj[j]);
        }
    }
    const double t = block_sum(a, sh);
    if (threadIdx.x == 0) {
        ye_s = t * e.Ee[1];
        y[e.nc] = ye_s;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < e.nc; j += DT) y[j] = (y[j] - e.Eje[j] * ye_s) * e.iEjj[j];
    __syncthreads();
}

// t = s .* v - (A Z y)_i, or - (A^T Z y)_i; y: the coarse solution (df.y or a copy). Only an active row (df.act) has a nonzero A Z y: its fixed
// coefficients times its own group's constant and the one on the membrane's other side. (Forming it from
// the row's cross-region entries here made every warp that meets an active row pay for the longest of
// its entry loops: 126 us at 128^3, 104 us of it FP64 issue; now 82 us.)
__device__ __forceinline__ void defl_input(int64_t i, const double* v, const double* __restrict__ s,
                                           const DeflFuse& df, const double* y, double t[4]) {
    const double2* vp = reinterpret_cast<const double2*>(v + 4 * i);
    const double2* sp = reinterpret_cast<const double2*>(s + 4 * i);
    const int32_t a = df.act[i];
    const double2 v0 = vp[0], v1 = vp[1], s0 = sp[0], s1 = sp[1];
    t[0] = s0.x * v0.x;
    t[1] = s0.y * v0.y;
    t[2] = s1.x * v1.x;
    t[3] = s1.y * v1.y;
    if (a < 0) return;
    const double yo = y[i < df.N_i ? df.rgrp[i] : df.ext_group], yc = y[df.xgrp[a]];
    const double* c = df.C + 8 * (int64_t)a;
    for (int q = 0; q < 4; ++q) t[q] -= c[q] * yo + c[4 + q] * yc;
}

}  // namespace knp
