// Flexible GMRES(m), FP64, right-preconditioned by one V-cycle on P_0 (Section 4.2,
// Section 6.2: restart 30, x_0 = u_{n-1}).
//
// The Krylov space is built for the symmetrically scaled system
// S^-1 A S^-1 (S x) = S^-1 f with S^2 = diag(P_0), which evens out the concentration and
// potential rows (their magnitudes differ by orders of magnitude); the scaling is applied
// on the fly (SpMV row scale, V-cycle input scale), so the preconditioned directions
// z_j live in the unscaled solution space and x = x_0 + Z y directly. Orthogonalisation
// is classical Gram-Schmidt with one reorthogonalisation (CGS2) in three fused passes; the
// second pass is made only when the first removed nearly all of the new vector (REORTH_KEEP).
//
// Stopping test: the preconditioned residual, as in Section 6.2, measured in the scaled
// norm and relative to the iterate x_c the current restart cycle began from (x_0 for the
// first cycle; or, if that is smaller, to the correction of the cycle, which covers a cold
// start), for the concentrations and the potentials apart:
// ||S M^-1 r_k||_g <= rtol max(||S x_c||_g, ||S (x_k - x_c)||_g) for g in {c, phi}. A residual norm
// alone is blind to the per-cell constant of phi_i (the intracellular potential block is
// singular up to the small membrane mass), while M^-1 r approximates the error. For the
// FGMRES iterate, M^-1 r_k = Z_{k+1} c with c = Q_k^T g_k e_{k+1} from the Givens rotations,
// so its group S-norms (and those of the correction Z y_k) take one pass over Z. That pass is
// made only when the test may pass: each evaluation records est_g / |g_k|, and the next is
// scheduled once that ratio times the current Givens residual |g_k| comes near the threshold.
// (Apart, because the scaled concentrations outweigh the scaled potentials by two orders.)
// The host sees one Hessenberg column per iteration.
#include <sched.h>

#include <algorithm>
#include <chrono>
#include <map>
#include <memory>
#include <tuple>
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "deflate.h"
#include "gmres.h"
#include "problem.h"
#include "vcycle.h"

namespace knp {

namespace {

constexpr int RED_BLOCKS = 152;   // the most blocks a reduction kernel launches: one per SM (152 SMs)
constexpr int RED_THREADS = 256;  // the most threads of a block
constexpr int MAXV = 32;          // restart + 2
constexpr int MAXW = 3 * MAXV;    // the most sums a reduction kernel forms
constexpr int PART_LD = RED_BLOCKS + 8;   // partial[k * PART_LD + b]: block b's share of sum k
// device scalars: [0, MAXV) first-pass dots, [MAXV, 2 MAXV) second-pass dots, [2 MAXV, 2 MAXV +
// MAXW) reference norms, 2 MAXV + MAXW the skip flag, then the six stopping-test norms, then the
// second-pass flag of the Arnoldi step
constexpr int SKIP_OFF = 2 * MAXV + MAXW;
constexpr int CHK_OFF = SKIP_OFF + 1;
constexpr int SECOND_OFF = CHK_OFF + 6;
constexpr int DOTS_LEN = SECOND_OFF + 1;
constexpr int CHECK_EVERY = 8;         // steps between exact evaluations of the stopping test, at most
                                       // (8 against 4: 0.8-1.4% less time per step on the 3D and 2D
                                       // workloads, iteration counts equal or +2 in 290)
constexpr double CHECK_MARGIN = 10.0;  // evaluate once a prediction is within this factor of passing

// What bounds these kernels: an FP64 instruction holds an SM's FP64 pipe for 16 cycles per warp, so
// what counts is the number of warp instructions, not only the vector elements: a reduction's adds
// and any scalar that every thread works out for itself cost as much as vector work. Hence one block
// of 8 warps per SM whose threads take two elements (16 bytes) of each vector at a time, so that the
// 31 adds of a warp's reduction are paid by 8 warps per SM and not by 32; scalars are formed once per
// block; and each kernel sums the partial results of the one before it in its prologue (about 1 us)
// instead of a reduction launch (4.8 us) between them.
// Every kernel is instantiated for a compile-time vector count NV, so that the accumulators and
// basis values stay in registers (a runtime count put them on the stack).

// One halving step of a warp reduce-scatter of C values per lane (C even): lanes with bit O
// set keep the upper half and receive their partner's upper half, the others the lower half.
template <int C>
__device__ __forceinline__ void warp_halve(double* v, int lane, int O) {
    const bool hi = (lane & O) != 0;
#pragma unroll
    for (int k = 0; k < C / 2; ++k) {
        const double send = hi ? v[k] : v[k + C / 2];
        const double keep = hi ? v[k + C / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
}

// Warp sums of C values per lane (C a power of two up to 32): C - 1 adds of a reduce-scatter, then
// one for each halving of the lanes that are left. Returns the sum of value lane / (32 / C).
template <int C>
__device__ __forceinline__ double warp_sums(double* v, int lane) {
    if constexpr (C == 32) warp_halve<32>(v, lane, 16);
    if constexpr (C >= 16) warp_halve<16>(v, lane, C == 32 ? 8 : 16);
    if constexpr (C >= 8) warp_halve<8>(v, lane, C == 32 ? 4 : C == 16 ? 8 : 16);
    if constexpr (C >= 4) warp_halve<4>(v, lane, C == 32 ? 2 : C == 16 ? 4 : C == 8 ? 8 : 16);
    if constexpr (C >= 2) warp_halve<2>(v, lane, C == 32 ? 1 : C == 16 ? 2 : C == 8 ? 4 : C == 4 ? 8 : 16);
    double s = v[0];
#pragma unroll
    for (int o = 16 / C; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

template <int NT>
constexpr int POW2 = NT <= 1 ? 1 : NT <= 2 ? 2 : NT <= 4 ? 4 : NT <= 8 ? 8 : NT <= 16 ? 16 : 32;

// Block sums of NT values per thread (NT <= 32) into partial[k * PART_LD + blockIdx.x]
template <int NT>
__device__ __forceinline__ void block_reduce_store(const double (&acc)[NT], double* __restrict__ partial) {
    constexpr int C = POW2<NT>;
    static_assert(NT <= 32, "at most 32 sums");
    __shared__ double sh[RED_THREADS / 32][C];
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    double v[C];
#pragma unroll
    for (int k = 0; k < C; ++k) v[k] = k < NT ? acc[k] : 0.0;
    const double s = warp_sums<C>(v, lane);
    if (lane % (32 / C) == 0) sh[wid][lane / (32 / C)] = s;
    __syncthreads();
    if (threadIdx.x < NT) {
        double t = 0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) t += sh[w][threadIdx.x];
        partial[threadIdx.x * PART_LD + blockIdx.x] = t;
    }
}

// out[k] = sum over blocks of partial[k * PART_LD + b], k < nt, by one block: each
// warp takes four sums at a time. Every block of a kernel gets the same bits. out is shared memory.
__device__ __forceinline__ void sum_partials(const double* partial, int nblocks, int nt, double* out) {
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    for (int k0 = 4 * wid; k0 < nt; k0 += 4 * ((int)blockDim.x / 32)) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = lane; b < nblocks; b += 32) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (k0 + q < nt) v[q] += partial[(k0 + q) * PART_LD + b];
        }
        const double s = warp_sums<4>(v, lane);
        if (lane % 8 == 0 && k0 + lane / 8 < nt) out[k0 + lane / 8] = s;
    }
    __syncthreads();
}

// Two neighbouring elements of a vector; vectors are 4 n doubles, 16-byte aligned
__device__ __forceinline__ double2 ld2(const double* p, int64_t i2) {
    return reinterpret_cast<const double2*>(p)[i2];
}
__device__ __forceinline__ void st2(double* __restrict__ p, int64_t i2, double2 v) {
    reinterpret_cast<double2*>(p)[i2] = v;
}

// Pairs per thread and sweep: few vectors leave too few bytes in flight with one
template <int NV>
constexpr int PAIRS = NV <= 3 ? 4 : NV <= 7 ? 2 : 1;

// partial sums of <V_k, w> for k < NV, and of <w, w> at k = NV
template <int NV>
__global__ void __launch_bounds__(RED_THREADS, 1) k_mdot(int64_t n4, const double* V, int64_t ldv,
                                                         const double* w, double* __restrict__ partial) {
    chain_wait();
    constexpr int E = PAIRS<NV>;
    double acc[NV + 1];
#pragma unroll
    for (int k = 0; k <= NV; ++k) acc[k] = 0.0;
    const int64_t n2 = n4 / 2, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += E * stride) {
        double2 wi[E], vk[E][NV > 0 ? NV : 1];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool in = e == 0 || i + e * stride < n2;
            wi[e] = in ? ld2(w, i + e * stride) : make_double2(0.0, 0.0);
#pragma unroll
            for (int k = 0; k < NV; ++k) vk[e][k] = in ? ld2(V + k * ldv, i + e * stride) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e > 0 && i + e * stride >= n2) break;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                acc[k] += vk[e][k].x * wi[e].x;
                acc[k] += vk[e][k].y * wi[e].y;
            }
            acc[NV] += wi[e].x * wi[e].x;
            acc[NV] += wi[e].y * wi[e].y;
        }
    }
    block_reduce_store<NV + 1>(acc, partial);
}

// Sums of squares per group of an element-wise quantity: groups 0 = concentrations (fields 0..2), 1 =
// potentials (field 3); with NG = 3, group 2 takes the extracellular potentials (elements at or past
// n4i). A thread's pairs are all fields (0, 1) or all fields (2, 3), since the grid stride is even, and
// its potentials cross the region boundary at most once.
template <int NG>
struct GroupSums {
    double a = 0.0, b = 0.0, before = 0.0;   // first and second element of the pair; b up to the boundary
    bool past = false;
    __device__ __forceinline__ void add(int64_t i2, int64_t n4i, double x, double y) {
        if (NG == 3 && !past && 2 * i2 >= n4i) {
            before = b;
            b = 0.0;
            past = true;
        }
        a += x * x;
        b += y * y;
    }
    // out[0..NG): this thread's sums; hi: its pairs are fields (2, 3)
    __device__ __forceinline__ void get(bool hi, double* out) const {
        out[0] = hi ? a : a + (NG == 3 ? before + b : b);
        out[1] = !hi ? 0.0 : NG == 3 ? (past ? before : b) : b;
        if (NG == 3) out[NG - 1] = hi && past ? b : 0.0;
    }
};

// partial sums of ||s .* w||^2 per group (the stopping test's reference norms)
template <int NG>
__global__ void __launch_bounds__(RED_THREADS) k_group_norms(int64_t n4, const double* __restrict__ w,
                                                             const double* __restrict__ s, int64_t n4i,
                                                             double* __restrict__ partial) {
    GroupSums<NG> g;
    const int64_t n2 = n4 / 2, i0 = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x;
    for (int64_t i = i0; i < n2; i += (int64_t)gridDim.x * RED_THREADS) {
        const double2 wi = ld2(w, i), si = ld2(s, i);
        g.add(i, n4i, wi.x * si.x, wi.y * si.y);
    }
    double out[NG];
    g.get((i0 & 1) != 0, out);
    block_reduce_store<NG>(out, partial);
}

// Partial sums of the S^2-weighted squared norms, by group, of two combinations of the columns of Z:
// u = sum_k c[k] Z_k and v = sum_k y[k] Z_k (y[NV-1] is the newest column's, often 0).
// Slot g holds group g's part of ||u||_S^2 and slot NG + g that of ||v||_S^2 (groups as above).
// Without with_y only u is formed (v's slots are zero): half the FP64 work.
template <int NV, int NG>
__global__ void __launch_bounds__(RED_THREADS, 1) k_combo_norms(int64_t n4, const double* __restrict__ Z, int64_t ldz,
                                                                const double* __restrict__ cy,
                                                                const double* __restrict__ s, int64_t n4i,
                                                                double* __restrict__ partial, int with_y) {
    constexpr int E = PAIRS<NV>;
    __shared__ double ck[NV > 0 ? NV : 1], yk[NV > 0 ? NV : 1];
    if ((int)threadIdx.x < NV) {
        ck[threadIdx.x] = cy[threadIdx.x];
        yk[threadIdx.x] = cy[MAXV + threadIdx.x];
    }
    __syncthreads();
    GroupSums<NG> gu, gv;
    const int64_t n2 = n4 / 2, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < n2; i += E * stride) {
        double2 zk[E][NV > 0 ? NV : 1], w[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool in = e == 0 || i + e * stride < n2;
            w[e] = in ? ld2(s, i + e * stride) : make_double2(0.0, 0.0);
#pragma unroll
            for (int k = 0; k < NV; ++k) zk[e][k] = in ? ld2(Z + k * ldz, i + e * stride) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e > 0 && i + e * stride >= n2) break;
            double2 u = make_double2(0.0, 0.0);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                u.x += ck[k] * zk[e][k].x;
                u.y += ck[k] * zk[e][k].y;
            }
            gu.add(i + e * stride, n4i, u.x * w[e].x, u.y * w[e].y);
            if (with_y) {
                double2 v = make_double2(0.0, 0.0);
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    v.x += yk[k] * zk[e][k].x;
                    v.y += yk[k] * zk[e][k].y;
                }
                gv.add(i + e * stride, n4i, v.x * w[e].x, v.y * w[e].y);
            }
        }
    }
    double out[2 * NG];
    gu.get((i0 & 1) != 0, out);
    gv.get((i0 & 1) != 0, out + NG);
    block_reduce_store<2 * NG>(out, partial);
}

// w' = w - sum_k h[k] V_k (in place), h the sums of the first pass's partial dots (pdots); partial sums
// of <V_k, w'> and <w', w'>. Block 0 stores h to dots and the flag below to dots[SECOND_OFF]. When the
// first pass kept at least REORTH_KEEP of w's squared norm (|w'|^2 = <w,w> - |h|^2 >= REORTH_KEEP
// <w,w>), w' is orthogonal to the basis to about eps / sqrt(REORTH_KEEP) and the second pass is
// skipped: only <w', w'> is formed, and k_orth_final then just normalises. This is the
// Daniel-Gragg-Kaufman-Stewart test with a looser threshold than its usual 1/2: on the FGMRES
// workloads here the first pass keeps 8-20% of |w|^2, the second pass found nothing to remove in
// 85-99% of the steps, and FP64 issue (not bandwidth) bounds these kernels on GB300.
constexpr double REORTH_KEEP = 1e-4;
template <int NV>
__global__ void __launch_bounds__(RED_THREADS, 1) k_orth_update_dot(int64_t n4, const double* V,
                                                                    int64_t ldv, const double* pdots,
                                                                    int nblocks, double* __restrict__ dots, double* w,
                                                                    double* __restrict__ partial) {
    constexpr int E = PAIRS<NV>;
    __shared__ double h[NV + 1];
    __shared__ int second_s;
    chain_wait();
    sum_partials(pdots, nblocks, NV + 1, h);
    if (threadIdx.x == 0) {
        double hh = 0.0;
        for (int k = 0; k < NV; ++k) hh += h[k] * h[k];
        second_s = h[NV] - hh < REORTH_KEEP * h[NV];
        if (blockIdx.x == 0) dots[SECOND_OFF] = second_s ? 1.0 : 0.0;
    }
    if (blockIdx.x == 0 && threadIdx.x <= NV) dots[threadIdx.x] = h[threadIdx.x];
    __syncthreads();
    const bool second = second_s != 0;
    double hk[NV > 0 ? NV : 1];
#pragma unroll
    for (int k = 0; k < NV; ++k) hk[k] = h[k];
    const int64_t n2 = n4 / 2, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (second) {
        double acc[NV + 1];
#pragma unroll
        for (int k = 0; k <= NV; ++k) acc[k] = 0.0;
        for (int64_t i = i0; i < n2; i += stride) {
            double2 vk[NV > 0 ? NV : 1];
            double2 wi = ld2(w, i);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                vk[k] = ld2(V + k * ldv, i);
                wi.x -= hk[k] * vk[k].x;
                wi.y -= hk[k] * vk[k].y;
            }
            st2(w, i, wi);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                acc[k] += vk[k].x * wi.x;
                acc[k] += vk[k].y * wi.y;
            }
            acc[NV] += wi.x * wi.x;
            acc[NV] += wi.y * wi.y;
        }
        block_reduce_store<NV + 1>(acc, partial);
    } else {
        double acc[1] = {0.0};
        for (int64_t i = i0; i < n2; i += E * stride) {
            double2 wi[E], vk[E][NV > 0 ? NV : 1];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool in = e == 0 || i + e * stride < n2;
                wi[e] = in ? ld2(w, i + e * stride) : make_double2(0.0, 0.0);
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    vk[e][k] = in ? ld2(V + k * ldv, i + e * stride) : make_double2(0.0, 0.0);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e > 0 && i + e * stride >= n2) break;
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    wi[e].x -= hk[k] * vk[e][k].x;
                    wi[e].y -= hk[k] * vk[e][k].y;
                }
                st2(w, i + e * stride, wi[e]);
                acc[0] += wi[e].x * wi[e].x;
                acc[0] += wi[e].y * wi[e].y;
            }
        }
        block_reduce_store<1>(acc, partial + NV * PART_LD);
    }
}

// v = (w' - sum_k h2[k] V_k) / eta with eta^2 = <w',w'> - |h2|^2, h2 the sums of the second pass's
// partial dots (pdots; only <w', w'> without a second pass). When the second Gram-Schmidt pass found
// nothing to remove (|h2| <= ORTH_SKIP * |w'|), the subtraction is skipped, V is not read, eta = |w'|, and
// the host keeps h1 alone in the Hessenberg column (skip flag).
// Further blocks work beside those: ga.nchunks + ga.next of them form the coarse correction's partial sums
// of Z^T (s .* v) from w', and the last one sends the step's scalars to the host (host: pinned memory, laid
// out as dots, then the arrival flag). A gather kernel and a copy node of their own took their time in the
// chain before the next V-cycle. With the coarse solve in the V-cycle's first kernel as well, three steps of
// 4,612 unknowns in 2D take 2.87 ms instead of 3.00, of 117,504 in 3D 9.79 instead of 10.00.
constexpr double ORTH_SKIP = 1e-10;
template <int NV>
__global__ void __launch_bounds__(RED_THREADS) k_orth_final(int64_t n4, const double* V, int64_t ldv,
                                                            const double* pdots, int nblocks, const double* dots,
                                                            const double* w, double* v, double* host,
                                                            GatherArgs ga, const double* __restrict__ s) {
    static_assert(RED_THREADS == DT, "the gather's blocks");
    __shared__ double h2[NV + 1];
    __shared__ double inv_s;
    __shared__ int skip_s;
    chain_wait();
    const bool second = dots[SECOND_OFF] != 0.0;
    if (second) {
        sum_partials(pdots, nblocks, NV + 1, h2);
    } else {
        if ((int)threadIdx.x < NV) h2[threadIdx.x] = 0.0;
        sum_partials(pdots + NV * PART_LD, nblocks, 1, h2 + NV);
    }
    if (threadIdx.x == 0) {
        const double s2 = h2[NV];
        double hh = 0.0;
        if (second)
            for (int k = 0; k < NV; ++k) hh += h2[k] * h2[k];
        const bool skip = hh <= ORTH_SKIP * ORTH_SKIP * s2;
        const double e2 = skip ? s2 : s2 - hh;
        inv_s = e2 > 0 ? rsqrt(e2) : 0.0;
        skip_s = skip;
    }
    __syncthreads();
    const double inv_eta = inv_s;
    const bool skip = skip_s != 0;
    if (blockIdx.x == gridDim.x - 1) {
        volatile double* out = host;
        for (int k = threadIdx.x; k < DOTS_LEN; k += RED_THREADS)
            out[k] = k >= MAXV && k <= MAXV + NV ? h2[k - MAXV] : k == SKIP_OFF ? (skip ? 1.0 : 0.0) : dots[k];
        __threadfence_system();
        __syncthreads();
        if (threadIdx.x == 0) *reinterpret_cast<volatile uint64_t*>(host + DOTS_LEN) = 1;
        return;
    }
    const int ng = ga.nchunks + ga.next, nvec = (int)gridDim.x - 1 - ng;
    if ((int)blockIdx.x >= nvec) {
        __shared__ double sh[DT / 32];
        const double t = block_sum(gather_share(ga, (int)blockIdx.x - nvec,
                                                [&](int64_t i) {
                                                    double wi = w[i];
                                                    if (!skip)
                                                        for (int k = 0; k < NV; ++k) wi -= h2[k] * V[k * ldv + i];
                                                    return s[i] * (wi * inv_eta);
                                                }),
                                   sh);
        if (threadIdx.x == 0) ga.part[(int)blockIdx.x - nvec] = t;
        return;
    }
    const int64_t n2 = n4 / 2, stride = (int64_t)nvec * RED_THREADS;
    const int64_t i0 = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x;
    if (skip) {
        for (int64_t i = i0; i < n2; i += 2 * stride) {
            const bool two = i + stride < n2;
            double2 a = ld2(w, i), b = two ? ld2(w, i + stride) : a;
            st2(v, i, make_double2(a.x * inv_eta, a.y * inv_eta));
            if (two) st2(v, i + stride, make_double2(b.x * inv_eta, b.y * inv_eta));
        }
    } else {
        for (int64_t i = i0; i < n2; i += stride) {
            double2 wi = ld2(w, i);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double2 vk = ld2(V + k * ldv, i);
                wi.x -= h2[k] * vk.x;
                wi.y -= h2[k] * vk.y;
            }
            st2(v, i, make_double2(wi.x * inv_eta, wi.y * inv_eta));
        }
    }
}

// out[k] = sum over blocks of partial[k * PART_LD + b] (one block)
__global__ void __launch_bounds__(RED_THREADS) k_reduce(const double* __restrict__ partial, int nblocks, int nv,
                                                        double* __restrict__ out) {
    __shared__ double sh[MAXW];
    sum_partials(partial, nblocks, nv, sh);
    if (threadIdx.x < nv) out[threadIdx.x] = sh[threadIdx.x];
}

// x += sum_k y[k] Z_k
template <int NZ>
__global__ void __launch_bounds__(RED_THREADS) k_update_x(int64_t n4, const double* __restrict__ Z, int64_t ldz,
                                                          const double* __restrict__ y, double* __restrict__ x) {
    double yk[NZ > 0 ? NZ : 1];
#pragma unroll
    for (int k = 0; k < NZ; ++k) yk[k] = y[k];
    const int64_t n2 = n4 / 2;
    for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n2; i += (int64_t)gridDim.x * RED_THREADS) {
        double2 s = ld2(x, i);
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
            const double2 z = ld2(Z + k * ldz, i);
            s.x += yk[k] * z.x;
            s.y += yk[k] * z.y;
        }
        st2(x, i, s);
    }
}

// Blocks of a reduction kernel: one per SM, fewer when a block's threads would not have two pairs each.
// (Partial sums of more blocks cost more in the next kernel's prologue than the added warps gain.)
int red_grid(int64_t n4) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(RED_BLOCKS, (n4 + 4 * RED_THREADS - 1) / (4 * RED_THREADS)));
}
// The same for the Arnoldi step's dots and the stopping test (least: 64 threads) and the update (128, for its
// prologue's sums), in smaller blocks where 256 threads would not have a pair each on every SM: a block
// reduction costs a warp as much as a pair of elements, so a small vector goes to more SMs and fewer warps.
// Three steps of 4,612 unknowns in 2D 2.88 -> 2.62 ms, of the Kir problem on 97x75 7.16 -> 6.77. Smaller
// blocks at up to two pairs per thread made 117,504 unknowns in 3D 0.3% slower, everywhere 128^3 12%.
struct RedShape {
    int blocks, threads;
};
RedShape red_shape(int64_t n4, int least) {
    const int64_t n2 = n4 / 2;
    int t = RED_THREADS;
    while (t > least && n2 < (int64_t)RED_BLOCKS * t) t /= 2;
    if (t == RED_THREADS) return {red_grid(n4), t};
    return {(int)std::max<int64_t>(1, std::min<int64_t>(RED_BLOCKS, (n2 + t - 1) / t)), t};
}
// Blocks of a kernel that leaves no partial sums: two pairs per thread, up to four blocks per SM
unsigned vec_grid(int64_t n4) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(608, (n4 + 4 * RED_THREADS - 1) / (4 * RED_THREADS)));
}

#define KNP_NV_CASES(X) \
    X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16) X(17) X(18) X(19) \
    X(20) X(21) X(22) X(23) X(24) X(25) X(26) X(27) X(28) X(29) X(30) X(31)

#define KNP_NV_CASE_k_mdot(N) case N: launch(k_mdot<N>, rs.blocks, rs.threads, q, KNP_ARGS); break;
#define KNP_NV_CASE_k_combo_norms2(N) case N: k_combo_norms<N, 2><<<rs.blocks, rs.threads, 0, st>>>(KNP_ARGS); break;
#define KNP_NV_CASE_k_combo_norms3(N) case N: k_combo_norms<N, 3><<<rs.blocks, rs.threads, 0, st>>>(KNP_ARGS); break;
#define KNP_NV_CASE_k_orth_update_dot(N) case N: launch(k_orth_update_dot<N>, us.blocks, us.threads, q, KNP_ARGS); break;
#define KNP_NV_CASE_k_orth_final(N) case N: launch(k_orth_final<N>, nb_vec + ga.nchunks + ga.next + 1, RED_THREADS, q, KNP_ARGS); break;
#define KNP_NV_CASE_k_update_x(N) case N: k_update_x<N><<<nb_vec, RED_THREADS, 0, st>>>(KNP_ARGS); break;
// Launch KERNEL<nv> for a runtime nv in [0, 31], with the caller's grid: rs or us (RedShape), or nb_vec
#define KNP_LAUNCH_NV(nv, KERNEL)                                                                    \
    do {                                                                                             \
        switch (nv) {                                                                                \
            KNP_NV_CASES(KNP_NV_CASE_##KERNEL)                                                       \
            default: KNP_FAIL(KNP_ERR_INVALID_ARG, "vector count %d out of range", (int)(nv));        \
        }                                                                                            \
    } while (0)

__global__ void k_scale_copy(int64_t n4, const double* __restrict__ a, const double* __restrict__ s,
                             double* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n4) out[i] = a[i] * s[i];
}

__global__ void k_scale_inplace(int64_t n4, double* __restrict__ v, double s) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n4) v[i] *= s;
}

}  // namespace

struct GmresWork {
    int restart = 0;
    int64_t n4 = 0;
    DArray<double> V, Z, partial, dots, y, cy, tmp;
    DArray<double> ones;            // unit weights (the paper's unscaled stopping test), on first use
    double* hh = nullptr;           // pinned: the step's scalars as the device sends them (DOTS_LEN), arrival flag
    uint64_t* flag() { return reinterpret_cast<uint64_t*>(hh + DOTS_LEN); }
    // An iteration as a CUDA graph per (basis index j, transposed, w formed by the V-cycle, tail): the
    // Arnoldi step (operator product, the three orthogonalisation passes) and, with a tail, the
    // preconditioning of its result. The tail's kernels belong to the hierarchy that the graphs were
    // captured with.
    enum Tail { NO_TAIL, VCYCLE, DEFLATED_VCYCLE };
    struct Graph {
        cudaGraphExec_t exec = nullptr;
        int launches = 0;
    };
    std::map<std::tuple<int, bool, bool, int>, Graph> graphs;
    uint64_t graphs_amg = 0;        // AmgHierarchy::id of that hierarchy
    cudaStream_t cap = nullptr;     // capture stream (the problem's stream may be the legacy one)
    void drop_graphs() {
        for (auto& kv : graphs) cudaGraphExecDestroy(kv.second.exec);
        graphs.clear();
    }
    // partial sums: of an Arnoldi step's two passes, each read by the kernel after it, and the others'
    double* pass1() { return partial.p; }
    double* pass2() { return partial.p + MAXW * PART_LD; }
    double* other() { return partial.p + 2 * MAXW * PART_LD; }
    ~GmresWork() {
        drop_graphs();
        if (cap) cudaStreamDestroy(cap);
        if (hh) cudaFreeHost(hh);
    }
};

GmresWork* gmres_work(knp_problem* p, int restart) {
    if (p->gw && p->gw->restart == restart) return p->gw;
    delete p->gw;
    p->gw = nullptr;
    auto g = std::make_unique<GmresWork>();   // the problem's once it is whole: an allocation may fail
    g->restart = restart;
    g->n4 = 4 * p->n_nodes;
    g->V.alloc((restart + 1) * g->n4);
    g->Z.alloc((restart + 1) * g->n4);
    g->partial.alloc(3 * MAXW * PART_LD);   // first pass, second pass, everything else
    g->dots.alloc(DOTS_LEN);
    g->y.alloc(MAXV);
    g->cy.alloc(2 * MAXV);
    g->tmp.alloc(g->n4);
    KNP_CUDA(cudaMallocHost(&g->hh, DOTS_LEN * sizeof(double) + sizeof(uint64_t)));
    p->gw = g.release();
    return p->gw;
}

void gmres_free(GmresWork* g) { delete g; }

// squared norm of a device vector (through the multi-dot kernels)
static double norm2_dev(GmresWork& g, const double* v, cudaStream_t st) {
    count_launch(2);
    const int nb = red_grid(g.n4);
    k_mdot<0><<<nb, RED_THREADS, 0, st>>>(g.n4, nullptr, 0, v, g.other());
    k_reduce<<<1, RED_THREADS, 0, st>>>(g.other(), nb, 1, g.dots.p);
    double s;
    KNP_CUDA(cudaMemcpyAsync(&s, g.dots.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    KNP_CUDA(cudaStreamSynchronize(st));
    return s;
}

// w = S^-1 A z_j, into V_{j+1} orthogonalised against V_0..V_j (CGS2, second pass skipped on the
// device when it has nothing to remove) and normalised; the dots of both passes land in g.dots
static void arnoldi_kernels(knp_problem* p, GmresWork& g, int j, bool transpose, bool w_ready, const GatherArgs& ga,
                            const Queue& q) {
    const int64_t n4 = g.n4;
    const int nv = j + 1;
    const RedShape rs = red_shape(n4, 64), us = red_shape(n4, 128);
    const unsigned nb_vec = vec_grid(n4);
    double* zj = g.Z.p + (int64_t)j * n4;
    // not in place where the gather reads w beside the normalisation; else in place, which keeps one vector
    // less in the L2 cache (0.5% of a pass at 75^3)
    double* v1 = g.V.p + nv * n4;
    double* w = ga.part ? g.tmp.p : v1;
    op_apply(p, zj, w, p->sinv.p, nullptr, transpose, q, w_ready);
    ProfScope ps(&p->prof, KC_ORTHO, q.st);
    count_launch(3);
#define KNP_ARGS n4, g.V.p, n4, w, g.pass1()
    KNP_LAUNCH_NV(nv, k_mdot);
#undef KNP_ARGS
#define KNP_ARGS n4, g.V.p, n4, g.pass1(), rs.blocks, g.dots.p, w, g.pass2()
    KNP_LAUNCH_NV(nv, k_orth_update_dot);
#undef KNP_ARGS
#define KNP_ARGS n4, g.V.p, n4, g.pass2(), us.blocks, g.dots.p, w, v1, g.hh, ga, p->svec.p
    KNP_LAUNCH_NV(nv, k_orth_final);
#undef KNP_ARGS
    KNP_CUDA(cudaGetLastError());
}

// The iteration's graph (GmresWork::graphs), captured at first use; tail launches the kernels that
// precondition v_{j+1} into the queue it is given. One launch replaces some 20, the kernels' prologues
// overlap (launch.h), and the host has the step's scalars while the V-cycle runs. Graphs of the Arnoldi
// step (ending in a copy node) and the V-cycle with the coarse correction's two kernels between them left
// four gaps per iteration: three steps of the 2D problem with 4,612 unknowns took 3.73 ms, now 3.03; two
// of 64^3 27.0 and 26.1.
template <class TailFn>
static void iteration_graph_launch(knp_problem* p, GmresWork& g, int j, bool transpose, bool w_ready,
                                   GmresWork::Tail kind, TailFn&& tail) {
    if (g.graphs_amg != p->amg->id) {
        g.drop_graphs();
        g.graphs_amg = p->amg->id;
    }
    auto key = std::make_tuple(j, transpose, w_ready, (int)kind);
    auto it = g.graphs.find(key);
    if (it == g.graphs.end()) {
        if (!g.cap) KNP_CUDA(cudaStreamCreateWithFlags(&g.cap, cudaStreamNonBlocking));
        const int64_t before = g_launches.load();
        const Queue q(g.cap, true);
        KNP_CUDA(cudaStreamBeginCapture(g.cap, cudaStreamCaptureModeThreadLocal));
        try {
            arnoldi_kernels(p, g, j, transpose, w_ready,
                            kind == GmresWork::DEFLATED_VCYCLE && deflation_gather_beside(p) ? deflation_gather(p)
                                                                                             : GatherArgs{},
                            q);
            if (kind != GmresWork::NO_TAIL) tail(q);
        } catch (...) {
            cudaGraph_t tmp = nullptr;
            cudaStreamEndCapture(g.cap, &tmp);
            if (tmp) cudaGraphDestroy(tmp);
            throw;
        }
        cudaGraph_t graph = nullptr;
        KNP_CUDA(cudaStreamEndCapture(g.cap, &graph));
        GmresWork::Graph ng;
        ng.launches = (int)(g_launches.load() - before);
        g_launches.fetch_sub(ng.launches);
        cudaError_t e = cudaGraphInstantiate(&ng.exec, graph, 0);
        cudaGraphDestroy(graph);
        KNP_CUDA(e);
        it = g.graphs.emplace(key, ng).first;
    }
    KNP_CUDA(cudaGraphLaunch(it->second.exec, p->stream));
    count_launch(it->second.launches);
}

// Whether a wait for the GPU gives its core to other threads (cudaDeviceScheduleYield)
static bool waits_yield() {
    unsigned flags = 0;
    KNP_CUDA(cudaGetDeviceFlags(&flags));
    return (flags & cudaDeviceScheduleMask) == cudaDeviceScheduleYield;
}

// Waits until the device has sent the scalars of the Arnoldi step launched last. A failed launch or kernel
// ends the wait with its error. With `yield` it gives the core away between two looks, as CUDA's own waits
// do under that policy: beside a busy process on the same core, steps of 64^3 then take 0.3% of the core;
// looking on regardless took 28%.
static void wait_scalars(GmresWork& g, cudaStream_t st, bool yield) {
    const int64_t query_every = yield ? 16 : 4096;
    for (int64_t k = 1; !__atomic_load_n(g.flag(), __ATOMIC_ACQUIRE); ++k) {
        if (yield) sched_yield();
        if (k % query_every) continue;
        const cudaError_t e = cudaStreamQuery(st);
        if (e == cudaErrorNotReady) continue;
        KNP_CUDA(e);
        KNP_REQUIRE(__atomic_load_n(g.flag(), __ATOMIC_ACQUIRE), KNP_ERR_CUDA, "an Arnoldi step's scalars were not sent");
    }
}

knp_status_detail fgmres(knp_problem* p, const knp_solve_opts& o, knp_solve_stats& stats, double* x,
                         const double* fvec, bool transpose) {
    auto t0 = std::chrono::steady_clock::now();
    const int m = o.restart;
    KNP_REQUIRE(m >= 1 && m + 2 <= MAXV, KNP_ERR_INVALID_ARG, "restart must be in [1, %d]", MAXV - 2);
    GmresWork& g = *gmres_work(p, m);
    KNP_REQUIRE(p->amg, KNP_ERR_STATE, "knp_amg_setup has not been called");
    const int64_t inner0 = p->amg->inner_its;
    cudaStream_t st = p->stream;
    const int64_t n4 = g.n4;
    const unsigned nb = (unsigned)((n4 + 255) / 256);
    const bool paper_test = o.stop_test == KNP_TEST_PAPER;
    KNP_REQUIRE(o.stop_test == KNP_TEST_SCALED || paper_test, KNP_ERR_INVALID_ARG, "unknown stopping test %d",
                (int)o.stop_test);
    // the paper's test is one group over the whole vector: unit weights, no phi_e group
    const int NG = (o.phi_e_group && !paper_test) ? 3 : 2;
    const int64_t n4i = 4 * p->N_i;
    const bool defl = o.deflate != 0;
    if (defl) deflation_prepare(p);
    // the forward product of the preconditioner's result reads its w, which the V-cycle can form; the
    // Arnoldi step of z_j always follows its preconditioning directly
    const bool w_ready = !transpose && op_reads_w(p) && vcycle_forms_w(p);
    double* const wz = w_ready ? p->op_w.p : nullptr;
    auto precond = [&](const double* v, const double* s, double* z) {
        if (defl)
            deflated_precond_apply(p, v, s, z, transpose, wz);
        else
            precond_apply(p, v, s, z, wz);
    };
    if (paper_test && !g.ones.p) {
        g.ones.alloc(n4);
        std::vector<double> h(n4, 1.0);
        KNP_CUDA(cudaMemcpyAsync(g.ones.p, h.data(), n4 * sizeof(double), cudaMemcpyHostToDevice, st));
        KNP_CUDA(cudaStreamSynchronize(st));
    }
    const double* wts = paper_test ? g.ones.p : p->swt.p;
    const int nb_red = red_grid(n4);
    const RedShape rs = red_shape(n4, 64);
    const unsigned nb_vec = vec_grid(n4);
    // iterations from CUDA graphs, unless a kernel class is being profiled (event pairs go
    // around single launches) or graphs are switched off for the V-cycle as well; CG(P_0) waits for the
    // host in every application and stays outside
    const bool use_graphs = p->amg->use_graphs && p->prof.active < 0;
    const GmresWork::Tail tail_kind = p->amg->inner_cg_max_it > 0 ? GmresWork::NO_TAIL
                                      : defl                      ? GmresWork::DEFLATED_VCYCLE
                                                                  : GmresWork::VCYCLE;
    auto tail = [&](double* v, double* z, const Queue& q) {
        if (defl)
            deflated_vcycle_launch(p, v, p->svec.p, z, transpose, wz, q);
        else
            vcycle_launch(p, v, p->svec.p, z, DeflFuse{}, wz, q);
    };
    const bool yield = waits_yield();
    // reference norms of the stopping test, per group: ||S x|| of the iterate a cycle starts from
    // (the initial guess, then each restart's), taken together with the cycle's correction
    double tol[3] = {0, 0, 0};
    double paper_tol = 0.0;   // rtol ||M^-1 f||_2 (the paper's test)
    auto reference_norms = [&]() {
        if (paper_test) {
            tol[0] = tol[1] = paper_tol;
            return;
        }
        count_launch(2);
        if (NG == 3)
            k_group_norms<3><<<nb_red, RED_THREADS, 0, st>>>(n4, x, p->swt.p, n4i, g.other());
        else
            k_group_norms<2><<<nb_red, RED_THREADS, 0, st>>>(n4, x, p->swt.p, n4i, g.other());
        k_reduce<<<1, RED_THREADS, 0, st>>>(g.other(), nb_red, NG, g.dots.p + 2 * MAXV);
        double xn2[3] = {0, 0, 0};
        KNP_CUDA(cudaMemcpyAsync(xn2, g.dots.p + 2 * MAXV, NG * sizeof(double), cudaMemcpyDeviceToHost, st));
        KNP_CUDA(cudaStreamSynchronize(st));
        KNP_REQUIRE(std::isfinite(xn2[0]) && std::isfinite(xn2[1]) && std::isfinite(xn2[2]), KNP_ERR_NUMERIC,
                    "iterate is not finite");
        for (int q = 0; q < NG; ++q) tol[q] = o.rtol * std::sqrt(std::max(xn2[q], 0.0));
        if (NG == 3) {
            // phi_e is some 1e-8 of phi_i: below ~1e-14 of the whole potential the rounding of the
            // coupled equations sets the floor, and a tighter request would stagnate
            const double floor_rel = o.phi_e_floor > 0 ? o.phi_e_floor : 1e-14;
            tol[2] = std::max(tol[2], floor_rel * std::sqrt(std::max(xn2[1] + xn2[2], 0.0)));
        }
    };
    if (paper_test) {
        precond(fvec, g.ones.p, g.tmp.p);
        paper_tol = o.rtol * std::sqrt(norm2_dev(g, g.tmp.p, st));
        KNP_REQUIRE(std::isfinite(paper_tol), KNP_ERR_NUMERIC, "preconditioned right-hand side is not finite");
    }
    k_scale_copy<<<nb, 256, 0, st>>>(n4, fvec, p->sinv.p, g.tmp.p);
    count_launch();
    const double bnorm = std::sqrt(norm2_dev(g, g.tmp.p, st));
    KNP_REQUIRE(std::isfinite(bnorm), KNP_ERR_NUMERIC, "right-hand side is not finite");
    knp_status_detail res{KNP_OK, 0, 0, 0.0};
    // KNP_GMRES_MONITOR set: every iteration prints the stopping test's terms to stderr
    static const bool monitor = std::getenv("KNP_GMRES_MONITOR") != nullptr;
    std::vector<double> H((m + 1) * m), cs(m), sn(m), gv(m + 1), cyh(2 * MAXV);
    int its = 0, restarts = 0;
    bool converged = false;
    double beta = 0;
    while (!converged) {
        // V_0 = S^-1 (f - A x)
        op_apply(p, x, g.V.p, p->sinv.p, fvec, transpose);
        beta = std::sqrt(norm2_dev(g, g.V.p, st));
        KNP_REQUIRE(std::isfinite(beta), KNP_ERR_NUMERIC, "residual is not finite");
        if (beta == 0.0) {
            converged = true;
            break;
        }
        if (its >= o.max_it) break;
        if (its > 0) restarts++;
        reference_norms();
        count_launch();
        k_scale_inplace<<<nb, 256, 0, st>>>(n4, g.V.p, 1.0 / beta);
        std::fill(gv.begin(), gv.end(), 0.0);
        gv[0] = beta;
        int k_done = 0;   // Arnoldi steps whose Hessenberg columns are kept
        // The stopping test is evaluated exactly (one pass over Z) at the first step of a cycle,
        // at its last, at least every CHECK_EVERY steps, and whenever the group norms predicted
        // from the last evaluation (est_g scaled by the Givens residual |g_j|) come within
        // CHECK_MARGIN of their thresholds; convergence is only ever declared from an evaluation.
        double ratio[3] = {0, 0, 0}, corr_last[3] = {0, 0, 0};
        int last_check = -1;
        bool vc_queued = false;
        for (int j = 0; j <= m; ++j) {
            double* vj = g.V.p + (int64_t)j * n4;
            double* zj = g.Z.p + (int64_t)j * n4;
            // z_j = P_0^{-1} (S v_j) (one V-cycle, or CG(P_0)), unless the previous step queued it
            if (!vc_queued) precond(vj, p->svec.p, zj);
            vc_queued = false;
            const bool arnoldi = (j < m) && (its < o.max_it);
            bool check = last_check < 0 || !arnoldi || j - last_check >= CHECK_EVERY;
            if (!check) {
                check = true;
                for (int q = 0; q < NG; ++q) {
                    const double ref = std::max(tol[q], o.rtol * corr_last[q]);
                    if (ratio[q] * std::fabs(gv[j]) > CHECK_MARGIN * ref) check = false;
                }
            }
            if (check) {
                // preconditioned residual of the iterate after j steps: M^-1 r = Z c with
                // c = Q^T (0, .., 0, g_j); the correction of this cycle, x_j - x_c = Z y_j
                const int k = j;
                std::fill(cyh.begin(), cyh.end(), 0.0);
                double* c = cyh.data();
                double* yk = cyh.data() + MAXV;
                c[k] = gv[k];
                for (int i = k - 1; i >= 0; --i) {
                    double a = c[i], b = c[i + 1];
                    c[i] = cs[i] * a - sn[i] * b;
                    c[i + 1] = sn[i] * a + cs[i] * b;
                }
                for (int i = k - 1; i >= 0; --i) {
                    double sacc = gv[i];
                    for (int q2 = i + 1; q2 < k; ++q2) sacc -= H[i * m + q2] * yk[q2];
                    yk[i] = sacc / H[i * m + i];
                }
                KNP_CUDA(cudaMemcpyAsync(g.cy.p, cyh.data(), 2 * MAXV * sizeof(double), cudaMemcpyHostToDevice,
                                         st));
                count_launch(2);
                // the correction's norm enters the reference only where a group's ||S x_c|| is zero
                // (a cold start); otherwise max(||S x_c||, ||S (x - x_c)||) is the state's norm
                // for every realistic step, so Z y is formed only in the first case
                bool with_y = false;
                for (int q = 0; q < NG; ++q) with_y |= tol[q] == 0.0;
#define KNP_ARGS n4, g.Z.p, n4, g.cy.p, wts, n4i, g.other(), (int)with_y
                if (NG == 3)
                    KNP_LAUNCH_NV(j + 1, k_combo_norms3);
                else
                    KNP_LAUNCH_NV(j + 1, k_combo_norms2);
#undef KNP_ARGS
                k_reduce<<<1, RED_THREADS, 0, st>>>(g.other(), rs.blocks, 2 * NG, g.dots.p + CHK_OFF);
            }
            const int nv = j + 1;
            if (arnoldi) {
                // v_{j+1} is normalised on the device: its preconditioning is queued before the host
                // waits for this step's scalars, so the GPU works while the host does the Givens step
                double *v1 = g.V.p + (int64_t)(j + 1) * n4, *z1 = g.Z.p + (int64_t)(j + 1) * n4;
                __atomic_store_n(g.flag(), 0, __ATOMIC_RELEASE);
                if (use_graphs)
                    iteration_graph_launch(p, g, j, transpose, w_ready, tail_kind,
                                           [&](const Queue& q) { tail(v1, z1, q); });
                else
                    arnoldi_kernels(p, g, j, transpose, w_ready, GatherArgs{}, st);
                if (!use_graphs || tail_kind == GmresWork::NO_TAIL) precond(v1, p->svec.p, z1);
                vc_queued = true;
                wait_scalars(g, st, yield);
            } else {
                KNP_CUDA(cudaMemcpyAsync(g.hh, g.dots.p, DOTS_LEN * sizeof(double), cudaMemcpyDeviceToHost, st));
                KNP_CUDA(cudaStreamSynchronize(st));
            }
            KNP_CUDA(cudaGetLastError());
            if (check) {
                bool ok = true;
                if (monitor) std::fprintf(stderr, "fgmres%s it %d |g| %.3e", transpose ? "^T" : "", its, std::fabs(gv[j]));
                if (paper_test) {
                    // one group: ||M^-1 r||_2 over the whole vector against rtol ||M^-1 f||_2; the
                    // ratio predicts it from the Givens residual as for the scaled test
                    const double e0 = g.hh[CHK_OFF], e1 = g.hh[CHK_OFF + 1];
                    KNP_REQUIRE(std::isfinite(e0) && std::isfinite(e1), KNP_ERR_NUMERIC,
                                "preconditioned residual is not finite");
                    const double est = std::sqrt(std::max(e0 + e1, 0.0));
                    ok = est <= paper_tol;
                    ratio[0] = ratio[1] = gv[j] != 0.0 ? est / std::fabs(gv[j]) : 0.0;
                    corr_last[0] = corr_last[1] = 0.0;
                    if (monitor) std::fprintf(stderr, "  est %.3e tol %.3e", est, paper_tol);
                } else {
                    for (int q = 0; q < NG; ++q) {
                        const double est2 = g.hh[CHK_OFF + q], corr2 = g.hh[CHK_OFF + NG + q];
                        KNP_REQUIRE(std::isfinite(est2) && std::isfinite(corr2), KNP_ERR_NUMERIC,
                                    "preconditioned residual is not finite");
                        const double est = std::sqrt(std::max(est2, 0.0)), corr = std::sqrt(std::max(corr2, 0.0));
                        const double ref = std::max(tol[q], o.rtol * corr);
                        ok &= est <= ref;
                        ratio[q] = gv[j] != 0.0 ? est / std::fabs(gv[j]) : 0.0;
                        corr_last[q] = corr;
                        if (monitor) std::fprintf(stderr, "  [%d] est %.3e tol %.3e corr %.3e", q, est, tol[q], corr);
                    }
                }
                if (monitor) std::fprintf(stderr, "\n");
                last_check = j;
                if (ok) {
                    converged = true;
                    k_done = j;
                    break;
                }
            }
            if (!arnoldi) {
                k_done = j;
                break;
            }
            // second pass skipped on the device (flag): the column is h1 and eta = |w'|
            const bool skipped = g.hh[SKIP_OFF] != 0.0;
            if (monitor) {
                // first Gram-Schmidt pass: |w'|^2 / |w|^2 = 1 - sum h1^2 / |w|^2
                double h1 = 0.0;
                for (int k = 0; k < nv; ++k) h1 += g.hh[k] * g.hh[k];
                std::fprintf(stderr, "arnoldi j %d pass1 ratio %.3e second-pass skipped %d\n", j,
                             g.hh[nv] > 0 ? 1.0 - h1 / g.hh[nv] : 0.0, (int)skipped);
            }
            double s2 = g.hh[MAXV + nv];
            double eta2 = s2;
            for (int k = 0; k < nv; ++k) {
                H[k * m + j] = g.hh[k] + (skipped ? 0.0 : g.hh[MAXV + k]);
                if (!skipped) eta2 -= g.hh[MAXV + k] * g.hh[MAXV + k];
            }
            KNP_REQUIRE(std::isfinite(eta2), KNP_ERR_NUMERIC, "Arnoldi vector is not finite");
            double eta = eta2 > 0 ? std::sqrt(eta2) : 0.0;
            H[(j + 1) * m + j] = eta;
            for (int k = 0; k < j; ++k) {
                double a = H[k * m + j], b = H[(k + 1) * m + j];
                H[k * m + j] = cs[k] * a + sn[k] * b;
                H[(k + 1) * m + j] = -sn[k] * a + cs[k] * b;
            }
            double den = std::hypot(H[j * m + j], H[(j + 1) * m + j]);
            cs[j] = H[j * m + j] / den;
            sn[j] = H[(j + 1) * m + j] / den;
            H[j * m + j] = den;
            H[(j + 1) * m + j] = 0.0;
            gv[j + 1] = -sn[j] * gv[j];
            gv[j] = cs[j] * gv[j];
            its++;
            k_done = j + 1;
            if (eta == 0.0) {
                converged = true;   // happy breakdown: the Krylov space holds the solution
                break;
            }
        }
        if (k_done > 0) {
            // y = R^-1 g (upper triangular), x += Z y
            std::vector<double> y(k_done);
            for (int k = k_done - 1; k >= 0; --k) {
                double s = gv[k];
                for (int q = k + 1; q < k_done; ++q) s -= H[k * m + q] * y[q];
                y[k] = s / H[k * m + k];
            }
            KNP_CUDA(cudaMemcpyAsync(g.y.p, y.data(), k_done * sizeof(double), cudaMemcpyHostToDevice, st));
            count_launch();
#define KNP_ARGS n4, g.Z.p, n4, g.y.p, x
            KNP_LAUNCH_NV(k_done, k_update_x);
#undef KNP_ARGS
            KNP_CUDA(cudaGetLastError());
        }
        if (!converged && its >= o.max_it) {
            res.code = KNP_ERR_NOT_CONVERGED;
            break;
        }
    }
    // report the scaled true residual of the final iterate
    op_apply(p, x, g.tmp.p, p->sinv.p, fvec, transpose);
    double rn = std::sqrt(norm2_dev(g, g.tmp.p, st));
    double relres = bnorm > 0 ? rn / bnorm : 0.0;
    if (!converged) res.code = KNP_ERR_NOT_CONVERGED;
    res.iterations = its;
    res.restarts = restarts;
    res.relres = relres;
    stats.iterations = its;
    stats.restarts = restarts;
    stats.inner_iterations = p->amg->inner_its - inner0;
    stats.true_relres = relres;
    stats.ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return res;
}

}  // namespace knp
