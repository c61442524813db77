// One V-cycle of the smoothed-aggregation hierarchy on P_0, the inexact P_0^{-1} of
// Section 4.2 (the paper uses one BoomerAMG V-cycle; here smoothed aggregation with
// Chebyshev smoothing, all four fields of a node in one pass). Templated on the
// storage/arithmetic type of the hierarchy: double (plain FP64 form) or float (the
// mixed-precision form; the coarsest dense solve is FP64 in both).
//
// Layouts: a level operator with short rows (the finest, about 15 entries per row in 3D) or
// with enough rows to fill the GPU one thread per row is sliced-ELL; the other operators and the
// restriction are CSR with 4 to 128 lanes per row; the prolongation is sliced-ELL over rows sorted by
// length. A lane always works on all four fields of an entry, so that the sums over a row's lanes can be
// a reduce-scatter and no lane of the slow FP64 pipe idles.
//
// Smoothing: Chebyshev steps on [lambda_max / ratio, 1.1 lambda_max] per field, `pre` of them
// before the coarse-grid correction (the first from x = 0 costs no operator product) and
// `degree` after; one before and two after by default, which makes the V-cycle non-symmetric
// (FGMRES takes any preconditioner; CG(P_0) is given as many steps before as after).
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <map>
#include <memory>
#include <mutex>
#include <type_traits>

#include "amg.h"
#include "amg_gpu.h"
#include "deflate_input.h"
#include "lanes.h"
#include "launch.h"
#include "problem.h"
#include "vcycle.h"

namespace knp {

namespace {

template <class T>
struct V4;
template <>
struct V4<double> {
    double v[4];
    __device__ __forceinline__ static V4 load(const double* p) {
        const double2* q = reinterpret_cast<const double2*>(p);
        double2 a = q[0], b = q[1];
        return V4{{a.x, a.y, b.x, b.y}};
    }
    __device__ __forceinline__ void store(double* p) const {
        double2* q = reinterpret_cast<double2*>(p);
        q[0] = make_double2(v[0], v[1]);
        q[1] = make_double2(v[2], v[3]);
    }
};
template <>
struct V4<float> {
    float v[4];
    __device__ __forceinline__ static V4 load(const float* p) {
        float4 a = *reinterpret_cast<const float4*>(p);
        return V4{{a.x, a.y, a.z, a.w}};
    }
    __device__ __forceinline__ void store(float* p) const {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};

struct Coef4 {
    double c1[4], c2[4];
};

__device__ __forceinline__ double pick4(const double c[4], int f) {
    return f == 0 ? c[0] : f == 1 ? c[1] : f == 2 ? c[2] : c[3];
}

// N consecutive fields of a node (4: one vector access)
template <class T, int N>
struct VN {
    T v[N];
    __device__ __forceinline__ static VN load(const T* p) {
        VN o;
        if constexpr (N == 4) {
            const V4<T> a = V4<T>::load(p);
#pragma unroll
            for (int f = 0; f < 4; ++f) o.v[f] = a.v[f];
        } else {
#pragma unroll
            for (int f = 0; f < N; ++f) o.v[f] = p[f];
        }
        return o;
    }
    __device__ __forceinline__ void store(T* p) const {
        if constexpr (N == 4) {
            V4<T>{{v[0], v[1], v[2], v[3]}}.store(p);
        } else {
#pragma unroll
            for (int f = 0; f < N; ++f) p[f] = v[f];
        }
    }
};

// Row product of a sliced-ELL operator by L lanes: lane t adds entries t, t + L, ... The loads of
// U entries (and the columns of the next batch) are issued together, so that a lane waits
// for memory once or twice per batch instead of twice per entry; the order of the sums is that of
// the entries. One thread per row: four entries in FP32, which memory bounds (two steps of the 125-cell
// 128^3 workload 228 -> 220 ms, most of it on the first coarse level's rows of 58 entries), one in FP64,
// which the FP64 pipe bounds (two entries cost registers and 1% at 64^3).
template <class T, int L>
__device__ __forceinline__ void sell_row(int64_t r, int t, const int64_t* __restrict__ sp,
                                         const int32_t* __restrict__ col, const T* __restrict__ val,
                                         const T* x, T acc[4]) {
    const int64_t s = r / SELL_C;
    const int64_t base = sp[s] + r % SELL_C;
    const int w = (int)((sp[s + 1] - sp[s]) / SELL_C);
    constexpr int U = L == 1 && sizeof(T) == 8 ? 1 : 4;
    const int32_t* cp = col + base;
    const T* vp = val + 4 * base;
    acc[0] = acc[1] = acc[2] = acc[3] = T(0);
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = t + u * L < w ? cp[(t + u * L) * SELL_C] : 0;
    chain_wait();
    for (int k = t; k < w; k += U * L) {
        V4<T> a[U], xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w) {
                a[u] = V4<T>::load(vp + 4 * ((k + u * L) * SELL_C));
                xv[u] = V4<T>::load(x + 4 * (int64_t)c[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = k + (U + u) * L;
            c[u] = q < w ? cp[q * SELL_C] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w)
                for (int f = 0; f < 4; ++f) acc[f] += a[u].v[f] * xv[u].v[f];
        }
    }
}

// Field t of a CSR row product by L lanes (t < L; lanes t < 4 of the row get the sum of field t): lane t
// takes entries t, t + L, ... with all four fields of each, CSR_BATCH<L> entries' loads in flight. Up to 32
// lanes are consecutive lanes of a warp; 128 lanes are the block, whose warps combine through shared
// memory. Blocks are 128 threads. Every thread of the block must call this (full-mask shuffles, and a
// block barrier for L = 128); rows r >= n pass active = false and contribute nothing.
// An FP64 instruction occupies the SM for 16 cycles whether 4 or 32 of its lanes do work. With all
// fields of an entry in one lane a row of n entries takes 4 ceil(n / L) instructions of 32 / L rows and
// 3 (L = 4) to 6 (L = 32) for the sums; one lane per field and entry slot took as many for a row's
// products and log2(slots) sums per row of half as many rows (64^3 FP64, 25,578 rows of 60 entries:
// Chebyshev step 26.6 -> 22.4 us; restriction to 235 rows of 600 entries 17.3 -> 8.3 us with a block
// per row).
template <int L>
constexpr int CSR_BATCH = L == 4 ? 2 : 4;   // many rows: registers for more blocks instead
template <class T, int L>
__device__ __forceinline__ T csr_row_field(bool active, int64_t r, int t, const int64_t* __restrict__ ptr,
                                           const int32_t* __restrict__ col, const T* __restrict__ val,
                                           const T* x) {
    static_assert(L == 4 || L == 8 || L == 16 || L == 32 || L == 128, "lanes per row");
    constexpr int U = CSR_BATCH<L>;
    T acc[4] = {T(0), T(0), T(0), T(0)}, out[1];
    const int64_t t0 = active ? ptr[r] + t : 0, t1 = active ? ptr[r + 1] : 0;
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = t0 + u * L < t1 ? col[t0 + u * L] : 0;
    chain_wait();
    if (active) {
        for (int64_t q = t0; q < t1; q += U * L) {
            V4<T> a[U], xv[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (q + u * L < t1) {
                    a[u] = V4<T>::load(val + 4 * (q + u * L));
                    xv[u] = V4<T>::load(x + 4 * (int64_t)c[u]);
                }
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = q + (U + u) * L < t1 ? col[q + (U + u) * L] : 0;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (q + u * L < t1)
                    for (int f = 0; f < 4; ++f) acc[f] += a[u].v[f] * xv[u].v[f];
        }
    }
    lane_reduce4<T, (L < 32 ? L : 32)>(acc, t, out);
    if constexpr (L == 128) {
        __shared__ T part[4][4];   // [warp][field]
        if ((threadIdx.x & 31) < 4) part[threadIdx.x >> 5][threadIdx.x & 3] = out[0];
        __syncthreads();
        const int f = threadIdx.x & 3;
        out[0] = (part[0][f] + part[1][f]) + (part[2][f] + part[3][f]);
    }
    return out[0];
}

// first Chebyshev step from x = 0: d = c2 D^-1 b, x = d (d stored if a second step reads it). On the finest level b = s .* v (double
// input), or s .* v - A Z y inside the coarse correction (df.y set), whose y it forms itself with SOLVE (block
// 0 keeps it for the last kernel). Blocks of DT threads.
template <class T, bool SOLVE>
__global__ void __launch_bounds__(DT) k_cheb_first(int64_t n, const double* v, const double* __restrict__ s, T* b,
                             const T* __restrict__ dinv, Coef4 c, T* __restrict__ x, T* __restrict__ d, DeflFuse df,
                             int write_d) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    V4<T> di = V4<T>::load(dinv + 4 * (i < n ? i : 0)), dd;
    chain_wait();
    const double* y = df.y;
    if constexpr (SOLVE) {
        __shared__ double ys[SOLVE_CELLS];
        coarse_solve(df.e, ys);
        if (blockIdx.x == 0 && (int)threadIdx.x <= df.e.nc) df.y[threadIdx.x] = ys[threadIdx.x];
        y = ys;
    }
    if (i >= n) return;
    V4<T> bb;
    if (v && df.y) {
        double t[4];
        defl_input(i, v, s, df, y, t);
        for (int f = 0; f < 4; ++f) bb.v[f] = (T)t[f];
        bb.store(b + 4 * i);
    } else if (v) {
        for (int f = 0; f < 4; ++f) bb.v[f] = (T)(s[4 * i + f] * v[4 * i + f]);
        bb.store(b + 4 * i);
    } else {
        bb = V4<T>::load(b + 4 * i);
    }
    for (int f = 0; f < 4; ++f) dd.v[f] = (T)c.c2[f] * di.v[f] * bb.v[f];
    if (write_d) dd.store(d + 4 * i);
    dd.store(x + 4 * i);
}

// Where the finest level's last smoothing step puts the V-cycle's result: z = x in FP64, every
// potential but the pinned one raised by its group's constant of the coarse correction (y set), and the
// operator product's w = sum_k z_k tau_r^k z^k (w set; needs all fields in one thread). Done there it
// saves a pass that reads x and one that reads z, and their launches.
struct VcycleOut {
    double* z = nullptr;
    double* w = nullptr;
    const double* y = nullptr;
    const int32_t* rgrp = nullptr;
    int64_t N_i = 0;
    int32_t pin = -1, ext_group = 0;
    double ztau[2][3] = {};
};

// fields f0 .. f0 + F of node i; lanes: with one field per lane, those of the warp that call this (a node's
// four neighbour each other), among which they form w
template <class T, int F>
__device__ __forceinline__ void store_out(const VcycleOut& o, int64_t i, int f0, const VN<T, F>& x, unsigned lanes = 0) {
    static_assert(F == 4 || F == 1, "a thread or a lane per field");
    VN<double, F> z;
    for (int f = 0; f < F; ++f) z.v[f] = (double)x.v[f];
    const bool in = i < o.N_i;
    if (o.y && f0 + F == 4 && i != o.pin) z.v[F - 1] += o.y[in ? o.rgrp[i] : o.ext_group];
    z.store(o.z + 4 * i + f0);
    if constexpr (F == 4) {
        if (o.w) {
            const double z0 = in ? o.ztau[0][0] : o.ztau[1][0], z1 = in ? o.ztau[0][1] : o.ztau[1][1],
                         z2 = in ? o.ztau[0][2] : o.ztau[1][2];
            o.w[i] = z0 * z.v[0] + z1 * z.v[1] + z2 * z.v[2];
        }
    } else {
        if (o.w && lanes) {
            const double zt = f0 == 0 ? o.ztau[in ? 0 : 1][0] : f0 == 1 ? o.ztau[in ? 0 : 1][1] : o.ztau[in ? 0 : 1][2];
            double w = f0 < 3 ? zt * z.v[0] : 0.0;
            w += __shfl_xor_sync(lanes, w, 1);
            w += __shfl_xor_sync(lanes, w, 2);
            if (f0 == 0) o.w[i] = w;
        }
    }
}

// Chebyshev step: r = b - A x_in; d = c1 d + c2 D^-1 r; x_out = x_in + d. The first step of a sweep
// (c1 = 0) does not read d, the last one does not store it; with OUT it is the V-cycle's last and writes
// its result instead of x_out.
template <class T, int L, bool OUT>
__global__ void __launch_bounds__(128) k_cheb_sell(int64_t n, const int64_t* __restrict__ sp,
                                                   const int32_t* __restrict__ col, const T* __restrict__ val,
                                                   const T* x_in, const T* b,
                                                   const T* __restrict__ dinv, Coef4 c, T* d,
                                                   T* __restrict__ x_out, int read_d, int write_d, VcycleOut out) {
    constexpr int F = LANE_FIELDS<L>;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = g / L;
    const int t = (int)(g % L);
    if (L == 1 && i >= n) return;   // with more lanes, all of a warp take part in the shuffles
    T acc[4], ax[F];
    sell_row<T, L>(i < n ? i : n - 1, t, sp, col, val, x_in, acc);
    lane_reduce4<T, L>(acc, t, ax);
    const unsigned lanes = OUT && L > 1 ? __ballot_sync(0xffffffffu, i < n && t < 4) : 0u;
    if (i >= n || t >= 4) return;
    const int f0 = lane_field<L>(t);
    const int64_t k = 4 * i + f0;
    VN<T, F> bb = VN<T, F>::load(b + k), di = VN<T, F>::load(dinv + k), xx = VN<T, F>::load(x_in + k), dd;
    if (read_d) {
        dd = VN<T, F>::load(d + k);
        for (int f = 0; f < F; ++f)
            dd.v[f] = (T)pick4(c.c1, f0 + f) * dd.v[f] + (T)pick4(c.c2, f0 + f) * di.v[f] * (bb.v[f] - ax[f]);
    } else {
        for (int f = 0; f < F; ++f) dd.v[f] = (T)pick4(c.c2, f0 + f) * di.v[f] * (bb.v[f] - ax[f]);
    }
    for (int f = 0; f < F; ++f) xx.v[f] += dd.v[f];
    if (write_d) dd.store(d + k);
    if constexpr (OUT)
        store_out<T, F>(out, i, f0, xx, lanes);
    else
        xx.store(x_out + k);
}

template <class T, int L, bool OUT>
__global__ void __launch_bounds__(128) k_cheb_csr(int64_t n, const int64_t* __restrict__ ptr,
                                                  const int32_t* __restrict__ col, const T* __restrict__ val,
                                                  const T* x_in, const T* b,
                                                  const T* __restrict__ dinv, Coef4 c, T* d,
                                                  T* __restrict__ x_out, int read_d, int write_d, VcycleOut out) {
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x), i = g / L;
    const int t = (int)(g % L);
    const T acc = csr_row_field<T, L>(i < n, i, t, ptr, col, val, x_in);
    if (t < 4 && i < n) {
        const int64_t k = 4 * i + t;
        T dd = (T)pick4(c.c2, t) * dinv[k] * (b[k] - acc);
        if (read_d) dd = (T)pick4(c.c1, t) * d[k] + dd;
        if (write_d) d[k] = dd;
        const T x = x_in[k] + dd;
        if constexpr (OUT)
            store_out<T, 1>(out, i, t, VN<T, 1>{{x}});
        else
            x_out[k] = x;
    }
}

// y = b - A x on a sliced-ELL level (b == nullptr: y = A x)
template <class T, int L>
__global__ void __launch_bounds__(128) k_resid_sell(int64_t n, const int64_t* __restrict__ sp,
                                                    const int32_t* __restrict__ col, const T* __restrict__ val,
                                                    const T* x, const T* b, T* __restrict__ y) {
    constexpr int F = LANE_FIELDS<L>;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = g / L;
    const int t = (int)(g % L);
    if (L == 1 && i >= n) return;
    T acc[4], ax[F];
    sell_row<T, L>(i < n ? i : n - 1, t, sp, col, val, x, acc);
    lane_reduce4<T, L>(acc, t, ax);
    if (i >= n || t >= 4) return;
    const int64_t k = 4 * i + lane_field<L>(t);
    VN<T, F> out;
    if (b) {
        out = VN<T, F>::load(b + k);
        for (int f = 0; f < F; ++f) out.v[f] -= ax[f];
    } else {
        for (int f = 0; f < F; ++f) out.v[f] = ax[f];
    }
    out.store(y + k);
}

template <class T, int L>
__global__ void __launch_bounds__(128) k_resid_csr(int64_t n, const int64_t* __restrict__ ptr,
                                                   const int32_t* __restrict__ col, const T* __restrict__ val,
                                                   const T* x, const T* b, T* __restrict__ r) {
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x), i = g / L;
    const int t = (int)(g % L);
    const T acc = csr_row_field<T, L>(i < n, i, t, ptr, col, val, x);
    if (t < 4 && i < n) r[4 * i + t] = b[4 * i + t] - acc;
}

// y = M x for a CSR with four values per entry (restriction)
template <class T, int L>
__global__ void __launch_bounds__(128) k_csr4(int64_t n, const int64_t* __restrict__ ptr,
                                              const int32_t* __restrict__ col, const T* __restrict__ val,
                                              const T* x, T* __restrict__ y) {
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x), i = g / L;
    const int t = (int)(g % L);
    const T acc = csr_row_field<T, L>(i < n, i, t, ptr, col, val, x);
    if (t < 4 && i < n) y[4 * i + t] = acc;
}

// x += P xc, P sliced ELL whose rows are sorted by length within windows (perm: sorted row -> row).
// One thread per row, or four (one per field) where that leaves too few threads: P's rows are short
// (about 6 entries), so splitting them over lanes would cost more in sums than it gains.
template <class T, int L>
__global__ void __launch_bounds__(128) k_prolong(int64_t n, const int64_t* __restrict__ sp,
                                                 const int32_t* __restrict__ col, const T* __restrict__ val,
                                                 const int32_t* __restrict__ perm, const T* xc, T* x) {
    static_assert(L == 1 || L == 4, "threads per row");
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t q = g / L;
    if (q >= n) return;
    const int64_t s = q / SELL_C, base = sp[s] + q % SELL_C;
    const int w = (int)((sp[s + 1] - sp[s]) / SELL_C);
    const int64_t r = perm[q];
    constexpr int U = L == 1 ? 2 : 4;
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = u < w ? col[base + u * SELL_C] : 0;
    chain_wait();
    if constexpr (L == 1) {
        V4<T> acc = V4<T>::load(x + 4 * r);
        for (int k0 = 0; k0 < w; k0 += U) {
            V4<T> a[U], v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + u < w) {
                    a[u] = V4<T>::load(val + 4 * (base + (k0 + u) * SELL_C));
                    v[u] = V4<T>::load(xc + 4 * (int64_t)c[u]);
                }
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = k0 + U + u < w ? col[base + (k0 + U + u) * SELL_C] : 0;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + u < w)
                    for (int f = 0; f < 4; ++f) acc.v[f] += a[u].v[f] * v[u].v[f];
        }
        acc.store(x + 4 * r);
    } else {
        const int f = (int)(g % L);
        T acc = x[4 * r + f];
        for (int k0 = 0; k0 < w; k0 += U) {
            T a[U], v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + u < w) {
                    a[u] = val[4 * (base + (k0 + u) * SELL_C) + f];
                    v[u] = xc[4 * (int64_t)c[u] + f];
                }
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = k0 + U + u < w ? col[base + (k0 + U + u) * SELL_C] : 0;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k0 + u < w) acc += a[u] * v[u];
        }
        x[4 * r + f] = acc;
    }
}

// x_f = Ainv_f b_f on the coarsest level, FP64; one warp per (field, row)
template <class T>
__global__ void k_coarse(int64_t nc, const double* __restrict__ inv, const T* b, T* __restrict__ x) {
    chain_wait();
    int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32;
    int lane = threadIdx.x % 32;
    if (wid >= 4 * nc) return;
    int f = (int)(wid / nc);
    int64_t row = wid % nc;
    const double* a = inv + ((int64_t)f * nc + row) * nc;
    double s = 0.0;
    for (int64_t j = lane; j < nc; j += 32) s += a[j] * (double)b[4 * j + f];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) x[4 * row + f] = (T)s;
}

template <class T>
__global__ void k_to_double(int64_t n4, const T* __restrict__ x, double* __restrict__ z) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n4) z[i] = (double)x[i];
}

// the V-cycle's result from x (a single-level hierarchy)
template <class T>
__global__ void k_out(int64_t n, const T* x, VcycleOut out) {
    chain_wait();
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n) store_out<T, 4>(out, r, 0, VN<T, 4>::load(x + 4 * r));
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <class T>
std::vector<T> cast_vec(const std::vector<double>& v) {
    return std::vector<T>(v.begin(), v.end());
}

// Lanes per row of the CSR kernels: 4, more (up to 32) while the grid stays below LANE_THREADS and a
// lane keeps two entries of a mean row; a block of 128 for few, very long rows (the restriction to the
// coarsest level: 235 rows of 600 entries at 64^3).
int csr_lanes(int64_t rows, double mean_len) {
    if (mean_len >= 256.0 && 128 * rows <= 2 * LANE_THREADS) return 128;
    int l = 4;
    while (l < 32 && 2 * l * rows <= LANE_THREADS && 4 * l <= mean_len) l *= 2;
    return l;
}

}  // namespace

template <class T>
__global__ void k_cast(int64_t n, const double* __restrict__ in, T* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = (T)in[i];
}

// device array of T from one of doubles: taken over as it is (T = double) or cast (T = float)
template <class T>
void take_values(DArray<T>& out, DArray<double>& in, int64_t count, cudaStream_t st) {
    if constexpr (std::is_same<T, double>::value) {
        out = std::move(in);
    } else {
        out.alloc(std::max<int64_t>(count, 1));
        if (count) k_cast<T><<<(unsigned)((count + 255) / 256), 256, 0, st>>>(count, in.p, out.p);
        KNP_CUDA(cudaStreamSynchronize(st));
        in.release();
    }
}

template <class T>
struct DevCsr4 {
    int64_t n = 0, nnz = 0;
    int lanes = 4;
    DArray<int64_t> ptr;
    DArray<int32_t> col;
    DArray<T> val;
    void upload(const HostCsr4& h, cudaStream_t st) {
        n = h.n_rows;
        nnz = h.nnz();
        lanes = csr_lanes(n, n ? (double)nnz / (double)n : 1.0);
        ptr.upload(h.ptr, st);
        col.upload(h.col, st);
        val.upload(cast_vec<T>(h.val), st);
    }
    // takes over a device CSR built by the GPU setup (no copy through the host)
    void take(DevCsr4d& d, cudaStream_t st) {
        n = d.n_rows;
        nnz = d.nnz;
        lanes = csr_lanes(n, n ? (double)nnz / (double)n : 1.0);
        ptr = std::move(d.ptr);
        col = std::move(d.col);
        take_values(val, d.val, 4 * d.nnz, st);
    }
};

// The prolongation as k_prolong reads it: sliced ELL over rows sorted by length, longest first, within
// windows of SORT_WINDOW rows. Unsorted, a warp runs as long as its longest row (P's rows have 1 to
// some 20 entries, about 6 on average), in FP64 instructions as in padding read; sorted over 256 rows the
// padding is a few percent and a window's writes still fall into the same lines (finest level at 64^3
// FP64 30.8 -> 22 us, at 128^3 FP32 115 -> 60 us).
constexpr int SORT_WINDOW = 256;

__global__ void __launch_bounds__(SORT_WINDOW) k_sort_rows(int64_t n, const int64_t* __restrict__ ptr,
                                                           int32_t* __restrict__ perm) {
    __shared__ int64_t len[SORT_WINDOW];
    const int64_t r = blockIdx.x * (int64_t)SORT_WINDOW + threadIdx.x;
    const int64_t mine = r < n ? ptr[r + 1] - ptr[r] : -1;
    len[threadIdx.x] = mine;
    __syncthreads();
    int rank = 0;
    for (int q = 0; q < SORT_WINDOW; ++q) rank += len[q] > mine || (len[q] == mine && q < (int)threadIdx.x);
    if (r < n) perm[blockIdx.x * (int64_t)SORT_WINDOW + rank] = (int32_t)r;
}

// entries of each slice of sorted rows: its first row is its longest
__global__ void k_sorted_widths(int64_t n, int64_t ns, const int64_t* __restrict__ ptr,
                                const int32_t* __restrict__ perm, int64_t* __restrict__ w) {
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const int64_t r = perm[s * SELL_C];
    w[s] = (ptr[r + 1] - ptr[r]) * SELL_C;
}

// CSR -> sorted sliced ELL; padding has zero values and repeats the row's last column (0 in an empty row)
template <class T>
__global__ void k_sorted_fill(int64_t n, int64_t ns, const int64_t* __restrict__ ptr, const int32_t* __restrict__ col,
                              const T* __restrict__ val, const int32_t* __restrict__ perm,
                              const int64_t* __restrict__ sp, int32_t* __restrict__ scol, T* __restrict__ sval) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= ns * SELL_C) return;
    const int64_t s = q / SELL_C, w = (sp[s + 1] - sp[s]) / SELL_C;
    const int64_t r = q < n ? perm[q] : -1;
    const int64_t len = r >= 0 ? ptr[r + 1] - ptr[r] : 0;
    for (int64_t k = 0; k < w; ++k) {
        const int64_t pos = sp[s] + q % SELL_C + k * SELL_C;
        scol[pos] = len > 0 ? col[ptr[r] + min(k, len - 1)] : 0;
        for (int f = 0; f < 4; ++f) sval[4 * pos + f] = k < len ? val[4 * (ptr[r] + k) + f] : T(0);
    }
}

template <class T>
struct DevProlong {
    int64_t n = 0;
    DArray<int64_t> sp;
    DArray<int32_t> col, perm;
    DArray<T> val;
    // builds the sorted form of P (whose CSR arrays can be released afterwards)
    void build(const DevCsr4<T>& P, cudaStream_t st) {
        n = P.n;
        if (!n) return;
        const int64_t ns = (n + SELL_C - 1) / SELL_C;
        perm.alloc(n);
        k_sort_rows<<<nblk(n, SORT_WINDOW), SORT_WINDOW, 0, st>>>(n, P.ptr.p, perm.p);
        DArray<int64_t> w;
        w.alloc(ns);
        k_sorted_widths<<<nblk(ns, 256), 256, 0, st>>>(n, ns, P.ptr.p, perm.p, w.p);
        sp.alloc(ns + 1);
        const int64_t total = device_exclusive_scan(w.p, sp.p, ns, st);
        col.alloc(std::max<int64_t>(total, 1));
        val.alloc(std::max<int64_t>(4 * total, 1));
        k_sorted_fill<T><<<nblk(ns * SELL_C, 128), 128, 0, st>>>(n, ns, P.ptr.p, P.col.p, P.val.p, perm.p, sp.p, col.p,
                                                                 val.p);
        KNP_CUDA(cudaStreamSynchronize(st));
    }
};

template <class T>
struct DevLevel {
    int64_t n = 0, nnz = 0;
    bool sell = false;
    int lanes = 1;   // lanes per row of the sliced-ELL kernels
    // sliced ELL (every level whose padding is small)
    DArray<int64_t> sp;
    DArray<int32_t> scol;
    DArray<T> sval;
    // CSR (levels too irregular for sliced ELL)
    DevCsr4<T> A;
    DArray<T> dinv;
    double lmax[4], lmin[4];
    DevProlong<T> P;
    DevCsr4<T> R;
    DArray<T> x, x2, b, r, d;
};

template <class T>
struct AmgDev {
    std::vector<std::unique_ptr<DevLevel<T>>> L;
    DArray<double> cinv;
    int64_t nc = 0;
    int degree = 2;                          // Chebyshev steps after the coarse-grid correction
    int pre = 1;                             // and before it (the first from x = 0: no operator product)
    std::vector<std::vector<Coef4>> coef;   // per level: coefficients of each Chebyshev step
};

static std::atomic<uint64_t> g_hierarchies{0};

AmgHierarchy::AmgHierarchy() : id(++g_hierarchies) {}

AmgHierarchy::~AmgHierarchy() {
    for (auto& kv : graphs)
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
    if (gstream) cudaStreamDestroy(gstream);
    delete static_cast<AmgDev<double>*>(h64);
    delete static_cast<AmgDev<float>*>(h32);
}

// A level's operator is stored sliced-ELL (one thread per row, the value loads of a warp
// contiguous) if its rows are short (at most SELL_SHORT_ROW entries on average), or if they are
// long but there are enough of them to keep the GPU busy with one thread each (at least
// SELL_MIN_LONG_ROWS); and in either case only if padding every slice to its longest row stores
// at most SELL_MAX_STORED entries per nonzero. Otherwise CSR with 4 to 128 lanes per row. Measured:
// the 512-cell 256^3 workload's first coarse level (1.7M rows of 58 entries) is 2.4% faster per
// FGMRES iteration as sliced ELL; P2's first coarse level at 32^3 (19.5k rows of 143 entries, four
// warps per SM with one thread per row) made the step 1.8 times slower.
constexpr double SELL_MAX_STORED = 2.0;
constexpr double SELL_SHORT_ROW = 24.0;
constexpr int64_t SELL_MIN_LONG_ROWS = 152 * 1024;

static bool sell_suits(int64_t rows, int64_t nnz) {
    return (double)nnz <= SELL_SHORT_ROW * (double)std::max<int64_t>(rows, 1) || rows >= SELL_MIN_LONG_ROWS;
}

// sliced ELL of a host CSR level; false (nothing done) if the level does not suit it (sell_suits,
// SELL_MAX_STORED)
template <class T>
static bool upload_sell(DevLevel<T>& L, const HostCsr4& A, cudaStream_t st) {
    const int64_t n = A.n_rows;
    int64_t ns = (n + SELL_C - 1) / SELL_C;
    std::vector<int64_t> sp(ns + 1, 0);
    for (int64_t s = 0; s < ns; ++s) {
        int64_t w = 0;
        for (int64_t r = s * SELL_C; r < std::min(n, (s + 1) * SELL_C); ++r) w = std::max(w, A.ptr[r + 1] - A.ptr[r]);
        sp[s + 1] = sp[s] + w * SELL_C;
    }
    if (!sell_suits(n, A.nnz()) || (double)sp[ns] > SELL_MAX_STORED * (double)std::max<int64_t>(A.nnz(), 1))
        return false;
    std::vector<int32_t> col(sp[ns]);
    std::vector<T> val(4 * sp[ns], T(0));
    for (int64_t s = 0; s < ns; ++s) {
        int64_t w = (sp[s + 1] - sp[s]) / SELL_C;
        for (int64_t lane = 0; lane < SELL_C; ++lane) {
            int64_t r = s * SELL_C + lane;
            int64_t len = r < n ? A.ptr[r + 1] - A.ptr[r] : 0;
            for (int64_t k = 0; k < w; ++k) {
                int64_t pos = sp[s] + k * SELL_C + lane;
                if (k < len) {
                    int64_t t = A.ptr[r] + k;
                    col[pos] = A.col[t];
                    for (int f = 0; f < 4; ++f) val[4 * pos + f] = (T)A.val[4 * t + f];
                } else {
                    col[pos] = (int32_t)std::min<int64_t>(r, n - 1);
                }
            }
        }
    }
    L.sp.upload(sp, st);
    L.scol.upload(col, st);
    L.sval.upload(val, st);
    return true;
}

// work vectors of a level and the coefficients of its Chebyshev steps (Saad's three-term
// recurrence on [lmin, lmax])
template <class T>
static void level_vectors_and_coefs(AmgDev<T>& D, DevLevel<T>& L, int degree, cudaStream_t st) {
    for (DArray<T>* v : {&L.x, &L.x2, &L.b, &L.r, &L.d}) {
        v->alloc(4 * L.n);
        v->zero(st);
    }
    std::vector<Coef4> cs(std::max(degree, 1));
    for (int f = 0; f < 4; ++f) {
        double th = 0.5 * (L.lmax[f] + L.lmin[f]), de = 0.5 * (L.lmax[f] - L.lmin[f]);
        double sigma = th / de;
        double rho0 = 1.0 / sigma;
        cs[0].c1[f] = 0.0;
        cs[0].c2[f] = 1.0 / th;
        for (int k = 1; k < degree; ++k) {
            double rho1 = 1.0 / (2.0 * sigma - rho0);
            cs[k].c1[f] = rho1 * rho0;
            cs[k].c2[f] = 2.0 * rho1 / de;
            rho0 = rho1;
        }
    }
    D.coef.push_back(cs);
}

template <class T>
static void upload_hierarchy(AmgDev<T>& D, const HostHierarchy& H, int degree, int pre, cudaStream_t st) {
    D.degree = degree;
    D.pre = pre;
    for (size_t l = 0; l < H.levels.size(); ++l) {
        const HostLevel& HL = H.levels[l];
        auto L = std::make_unique<DevLevel<T>>();
        const int64_t n = HL.A.n_rows;
        L->n = n;
        L->nnz = HL.A.nnz();
        L->sell = upload_sell(*L, HL.A, st);
        L->lanes = row_lanes(n, n ? (double)L->nnz / (double)n : 1.0);
        if (!L->sell) L->A.upload(HL.A, st);
        L->dinv.upload(cast_vec<T>(HL.dinv), st);
        for (int f = 0; f < 4; ++f) {
            L->lmax[f] = HL.lmax[f];
            L->lmin[f] = HL.lmin[f];
        }
        if (HL.P.n_rows) {
            DevCsr4<T> P;
            P.upload(HL.P, st);
            L->P.build(P, st);
            L->R.upload(HL.R, st);
        }
        level_vectors_and_coefs(D, *L, std::max(degree, pre), st);
        D.L.push_back(std::move(L));
    }
    D.nc = H.nc;
    D.cinv.upload(H.coarse_inv, st);
}

// sliced-ELL slice widths (entries per slice) from CSR row lengths
__global__ void k_sell_widths(int64_t n, int64_t ns, const int64_t* __restrict__ ptr, int64_t* __restrict__ w) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= ns) return;
    int64_t m = 0;
    for (int64_t r = s * SELL_C; r < min(n, (s + 1) * SELL_C); ++r) m = max(m, ptr[r + 1] - ptr[r]);
    w[s] = m * SELL_C;
}

// CSR -> sliced ELL; padding repeats the (clamped) row id with zero values, as upload_sell does
template <class T>
__global__ void k_sell_fill(int64_t n, int64_t ns, const int64_t* __restrict__ ptr, const int32_t* __restrict__ col,
                            const double* __restrict__ val, const int64_t* __restrict__ sp, int32_t* __restrict__ scol,
                            T* __restrict__ sval) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= ns * SELL_C) return;
    const int64_t s = r / SELL_C, lane = r % SELL_C;
    const int64_t w = (sp[s + 1] - sp[s]) / SELL_C;
    const int64_t len = r < n ? ptr[r + 1] - ptr[r] : 0;
    for (int64_t k = 0; k < w; ++k) {
        const int64_t pos = sp[s] + k * SELL_C + lane;
        if (k < len) {
            const int64_t t = ptr[r] + k;
            scol[pos] = col[t];
            for (int f = 0; f < 4; ++f) sval[4 * pos + f] = (T)val[4 * t + f];
        } else {
            scol[pos] = (int32_t)min(r, n - 1);
            for (int f = 0; f < 4; ++f) sval[4 * pos + f] = T(0);
        }
    }
}

// sliced ELL of a device CSR level (its CSR arrays released); false (nothing done) if the level
// does not suit it (sell_suits, SELL_MAX_STORED)
template <class T>
static bool take_sell(DevLevel<T>& L, DevCsr4d& A, cudaStream_t st) {
    const int64_t n = A.n_rows, ns = (n + SELL_C - 1) / SELL_C;
    if (!sell_suits(n, A.nnz)) return false;
    DArray<int64_t> w;
    w.alloc(std::max<int64_t>(ns, 1));
    k_sell_widths<<<nblk(ns, 256), 256, 0, st>>>(n, ns, A.ptr.p, w.p);
    DArray<int64_t> sp;
    sp.alloc(ns + 1);
    const int64_t total = device_exclusive_scan(w.p, sp.p, ns, st);
    if ((double)total > SELL_MAX_STORED * (double)std::max<int64_t>(A.nnz, 1)) return false;
    L.sp = std::move(sp);
    L.scol.alloc(std::max<int64_t>(total, 1));
    L.sval.alloc(std::max<int64_t>(4 * total, 1));
    k_sell_fill<T><<<nblk(ns * SELL_C, 128), 128, 0, st>>>(n, ns, A.ptr.p, A.col.p, A.val.p, L.sp.p, L.scol.p, L.sval.p);
    KNP_CUDA(cudaStreamSynchronize(st));
    A.ptr.release();
    A.col.release();
    A.val.release();
    return true;
}

// The same device hierarchy as upload_hierarchy, taken over from the GPU setup level by level
// (each level's setup arrays are released as soon as its V-cycle copy exists)
template <class T>
static void take_hierarchy(AmgDev<T>& D, GpuHierarchy& H, int degree, int pre, cudaStream_t st) {
    D.degree = degree;
    D.pre = pre;
    for (auto& G : H.levels) {
        auto L = std::make_unique<DevLevel<T>>();
        const int64_t n = G->A.n_rows;
        L->n = n;
        L->nnz = G->A.nnz;
        L->sell = take_sell(*L, G->A, st);
        L->lanes = row_lanes(n, n ? (double)L->nnz / (double)n : 1.0);
        if (!L->sell) L->A.take(G->A, st);
        take_values(L->dinv, G->dinv, 4 * n, st);
        for (int f = 0; f < 4; ++f) {
            L->lmax[f] = G->lmax[f];
            L->lmin[f] = G->lmin[f];
        }
        if (G->P.n_rows) {
            DevCsr4<T> P;
            P.take(G->P, st);
            L->P.build(P, st);
            L->R.take(G->R, st);
        }
        level_vectors_and_coefs(D, *L, std::max(degree, pre), st);
        D.L.push_back(std::move(L));
    }
    D.nc = H.nc;
    D.cinv.upload(H.coarse_inv, st);
}

void amg_upload(knp_problem* p, const HostHierarchy& H, int precision, int degree, int pre) {
    delete p->amg;
    p->amg = nullptr;
    auto amg = std::make_unique<AmgHierarchy>();   // the problem's once it is whole: an allocation may fail
    amg->precision = precision;
    amg->levels = (int)H.levels.size();
    amg->use_graphs = std::getenv("KNP_NO_GRAPHS") == nullptr;
    for (const HostLevel& L : H.levels) {
        amg->nodes.push_back(L.A.n_rows);
        amg->nnz.push_back(L.A.nnz());
    }
    if (precision == KNP_PREC_FP32) {
        auto* D = new AmgDev<float>();
        amg->h32 = D;
        upload_hierarchy(*D, H, degree, pre, p->stream);
    } else {
        auto* D = new AmgDev<double>();
        amg->h64 = D;
        upload_hierarchy(*D, H, degree, pre, p->stream);
    }
    KNP_CUDA(cudaStreamSynchronize(p->stream));
    p->amg = amg.release();
}

void amg_take_gpu(knp_problem* p, GpuHierarchy& H, int precision, int degree, int pre) {
    delete p->amg;
    p->amg = nullptr;
    auto amg = std::make_unique<AmgHierarchy>();   // the problem's once it is whole: an allocation may fail
    amg->precision = precision;
    amg->levels = (int)H.levels.size();
    amg->use_graphs = std::getenv("KNP_NO_GRAPHS") == nullptr;
    amg->setup_on_gpu = 1;
    amg->long_rows_p = H.long_rows_p;
    amg->long_rows_rap = H.long_rows_rap;
    for (auto& L : H.levels) {
        amg->nodes.push_back(L->A.n_rows);
        amg->nnz.push_back(L->A.nnz);
    }
    if (precision == KNP_PREC_FP32) {
        auto* D = new AmgDev<float>();
        amg->h32 = D;
        take_hierarchy(*D, H, degree, pre, p->stream);
    } else {
        auto* D = new AmgDev<double>();
        amg->h64 = D;
        take_hierarchy(*D, H, degree, pre, p->stream);
    }
    H.levels.clear();
    KNP_CUDA(cudaStreamSynchronize(p->stream));
    p->amg = amg.release();
}

// CSR kernels with the matrix's lanes per row
#define KNP_CSR_DISPATCH(lanes, KERNEL, rows, ...)                                                \
    switch (lanes) {                                                                              \
        case 4: launch(KERNEL(4), nblk((rows) * 4, 128), 128, q, __VA_ARGS__); break;             \
        case 8: launch(KERNEL(8), nblk((rows) * 8, 128), 128, q, __VA_ARGS__); break;             \
        case 16: launch(KERNEL(16), nblk((rows) * 16, 128), 128, q, __VA_ARGS__); break;          \
        case 32: launch(KERNEL(32), nblk((rows) * 32, 128), 128, q, __VA_ARGS__); break;          \
        default: launch(KERNEL(128), nblk((rows) * 128, 128), 128, q, __VA_ARGS__); break;        \
    }

// sliced-ELL kernels with the level's lanes per row
#define KNP_LANE_DISPATCH(lanes, KERNEL, rows, ...)                                               \
    switch (lanes) {                                                                              \
        case 1: launch(KERNEL(1), nblk(rows, 128), 128, q, __VA_ARGS__); break;                   \
        case 4: launch(KERNEL(4), nblk((rows) * 4, 128), 128, q, __VA_ARGS__); break;             \
        default: launch(KERNEL(8), nblk((rows) * 8, 128), 128, q, __VA_ARGS__); break;            \
    }
#define KNP_K_CHEB_SELL(L) k_cheb_sell<T, L, OUT>
#define KNP_K_CHEB_CSR(L) k_cheb_csr<T, L, OUT>
#define KNP_K_RESID_SELL(L) k_resid_sell<T, L>
#define KNP_K_RESID_CSR(L) k_resid_csr<T, L>
#define KNP_K_CSR4(L) k_csr4<T, L>

// Chebyshev step k of a sweep of `steps` steps; OUT: into `out` instead of x_out
template <class T, bool OUT = false>
static void launch_cheb(const DevLevel<T>& L, const T* x_in, const T* b, const Coef4& c, T* d, T* x_out, int k,
                        int steps, const Queue& q, const VcycleOut& out = VcycleOut{}) {
    count_launch();
    const int read_d = k > 0, write_d = k + 1 < steps;
    if (L.sell) {
        KNP_LANE_DISPATCH(L.lanes, KNP_K_CHEB_SELL, L.n, L.n, L.sp.p, L.scol.p, L.sval.p, x_in, b, L.dinv.p, c, d, x_out,
                          read_d, write_d, out);
    } else {
        KNP_CSR_DISPATCH(L.A.lanes, KNP_K_CHEB_CSR, L.n, L.n, L.A.ptr.p, L.A.col.p, L.A.val.p, x_in, b, L.dinv.p, c, d,
                         x_out, read_d, write_d, out);
    }
}

template <class T>
static void launch_resid(const DevLevel<T>& L, const T* x, const T* b, T* r, const Queue& q) {
    count_launch();
    if (L.sell) {
        KNP_LANE_DISPATCH(L.lanes, KNP_K_RESID_SELL, L.n, L.n, L.sp.p, L.scol.p, L.sval.p, x, b, r);
    } else {
        KNP_CSR_DISPATCH(L.A.lanes, KNP_K_RESID_CSR, L.n, L.n, L.A.ptr.p, L.A.col.p, L.A.val.p, x, b, r);
    }
}

template <class T>
static void cheb_step(DevLevel<T>& L, const Coef4& c, int k, int steps, Profiler* pr, bool fine, const Queue& q) {
    ProfScope ps(fine ? pr : nullptr, KC_CHEB_FINE, q.st);
    launch_cheb(L, L.x.p, L.b.p, c, L.d.p, L.x2.p, k, steps, q);
    std::swap(L.x.p, L.x2.p);
}

// the sweep's last step, whose result is the V-cycle's
template <class T>
static void cheb_step_out(DevLevel<T>& L, const Coef4& c, int k, int steps, const VcycleOut& out, Profiler* pr,
                          const Queue& q) {
    ProfScope ps(pr, KC_CHEB_FINE, q.st);
    launch_cheb<T, true>(L, L.x.p, L.b.p, c, L.d.p, nullptr, k, steps, q, out);
}

template <class T>
static void residual(DevLevel<T>& L, Profiler* pr, bool fine, const Queue& q) {
    ProfScope ps(fine ? pr : nullptr, KC_RESID_FINE, q.st);
    launch_resid(L, L.x.p, L.b.p, L.r.p, q);
}

// rc = R r
template <class T>
static void restrict_to(const DevCsr4<T>& R, const T* r, T* rc, const Queue& q) {
    count_launch();
    KNP_CSR_DISPATCH(R.lanes, KNP_K_CSR4, R.n, R.n, R.ptr.p, R.col.p, R.val.p, r, rc);
}

// x += P xc
template <class T>
static void prolong(const DevProlong<T>& P, const T* xc, T* x, const Queue& q) {
    count_launch();
    if (P.n >= LANE_THREADS)
        launch(k_prolong<T, 1>, nblk(P.n, 128), 128, q, P.n, P.sp.p, P.col.p, P.val.p, P.perm.p, xc, x);
    else
        launch(k_prolong<T, 4>, nblk(4 * P.n, 128), 128, q, P.n, P.sp.p, P.col.p, P.val.p, P.perm.p, xc, x);
}

template <class T>
static void smooth(DevLevel<T>& L, const std::vector<Coef4>& cs, int degree, bool zero_start, const double* v,
                   const double* s, const DeflFuse& df, Profiler* pr, bool fine, const Queue& q) {
    int k0 = 0;
    if (zero_start) {
        count_launch();
        launch(df.solve ? k_cheb_first<T, true> : k_cheb_first<T, false>, nblk(L.n, DT), DT, q, L.n, v, s, L.b.p,
               L.dinv.p, cs[0], L.x.p, L.d.p, df, degree > 1);
        k0 = 1;
    }
    for (int k = k0; k < degree; ++k) cheb_step(L, cs[k], k, degree, pr, fine, q);
}

template <class T>
static void vcycle_rec(AmgDev<T>& D, int l, const double* v, const double* s, const DeflFuse& df, Profiler* pr,
                       const Queue& q, const VcycleOut& out) {
    DevLevel<T>& L = *D.L[l];
    const int last = (int)D.L.size() - 1;
    if (l == last) {
        if (v) {
            // single-level hierarchy: build b from the scaled input first
            Coef4 c0{};
            count_launch();
            launch(df.solve ? k_cheb_first<T, true> : k_cheb_first<T, false>, nblk(L.n, DT), DT, q, L.n, v, s, L.b.p,
                   L.dinv.p, c0, L.x.p, L.d.p, df, 0);
        }
        count_launch();
        launch(k_coarse<T>, nblk(4 * D.nc * 32, 256), 256, q, D.nc, D.cinv.p, L.b.p, L.x.p);
        return;
    }
    DevLevel<T>& C = *D.L[l + 1];
    smooth(L, D.coef[l], D.pre, true, v, s, df, pr, l == 0, q);
    residual(L, pr, l == 0, q);
    restrict_to(L.R, L.r.p, C.b.p, q);
    vcycle_rec(D, l + 1, nullptr, nullptr, DeflFuse{}, pr, q, out);
    prolong(L.P, C.x.p, L.x.p, q);
    if (l > 0) {
        smooth(L, D.coef[l], D.degree, false, nullptr, nullptr, DeflFuse{}, pr, false, q);
    } else {
        for (int k = 0; k + 1 < D.degree; ++k) cheb_step(L, D.coef[l][k], k, D.degree, pr, true, q);
        cheb_step_out(L, D.coef[l][D.degree - 1], D.degree - 1, D.degree, out, pr, q);
    }
}

template <class T>
static void vcycle_typed(knp_problem* p, AmgDev<T>& D, const double* v, const double* s, double* z,
                         const DeflFuse& df, double* w, const Queue& q) {
    VcycleOut out;
    out.z = z;
    out.w = w;
    out.y = df.y;
    out.rgrp = df.rgrp;
    out.N_i = p->N_i;
    out.pin = df.pin;
    out.ext_group = df.ext_group;
    for (int r = 0; r < 2; ++r)
        for (int q = 0; q < 3; ++q) out.ztau[r][q] = p->sp.z[q] * p->sp.reg[r].tau[q];
    vcycle_rec(D, 0, v, s, df, &p->prof, q, out);
    if (D.L.size() == 1) {
        // no smoothing on a single level: the coarse solution is the result
        count_launch();
        launch(k_out<T>, nblk(D.L[0]->n, 256), 256, q, D.L[0]->n, D.L[0]->x.p, out);
    }
}

void vcycle_launch(knp_problem* p, const double* v, const double* s, double* z, const DeflFuse& df, double* w,
                   const Queue& q) {
    if (p->amg->h32)
        vcycle_typed(p, *static_cast<AmgDev<float>*>(p->amg->h32), v, s, z, df, w, q);
    else
        vcycle_typed(p, *static_cast<AmgDev<double>*>(p->amg->h64), v, s, z, df, w, q);
}

template <class T>
static bool forms_w(const AmgDev<T>& D) {
    return D.L.size() > 1 && D.L[0]->sell;
}

bool vcycle_forms_w(const knp_problem* p) {
    if (!p->amg || p->amg->inner_cg_max_it > 0) return false;
    return p->amg->h32 ? forms_w(*static_cast<AmgDev<float>*>(p->amg->h32))
                       : forms_w(*static_cast<AmgDev<double>*>(p->amg->h64));
}

void p0_apply(knp_problem* p, const double* x, double* y) {
    KNP_REQUIRE(p->amg && p->amg->h64, KNP_ERR_STATE, "P_0 products need the FP64 hierarchy");
    DevLevel<double>& L = *static_cast<AmgDev<double>*>(p->amg->h64)->L[0];
    KNP_REQUIRE(L.sell, KNP_ERR_STATE, "the finest level is not sliced ELL");
    launch_resid<double>(L, x, nullptr, y, p->stream);
    KNP_CUDA(cudaGetLastError());
}

// z = V-cycle(P_0)(s .* v); v, s, z are [n][4] doubles on the device. The V-cycle is a fixed
// sequence of about 15 launches, so it is captured once per set of arguments (AmgHierarchy::graphs)
// into a CUDA graph (on a private stream, since the problem's stream may be the legacy one) and
// replayed on the problem's stream. Each replay starts from
// scratch (the first kernel writes b, x and d of the finest level), so replays are independent.
// While a kernel class is being profiled, and with KNP_NO_GRAPHS, the launches go out one by one.
// (The V-cycles inside FGMRES iterations are parts of those iterations' graphs instead, gmres.cu.)
void vcycle_apply(knp_problem* p, const double* v, const double* s, double* z, const DeflFuse* dfp, double* w) {
    KNP_REQUIRE(p->amg, KNP_ERR_STATE, "knp_amg_setup has not been called");
    AmgHierarchy& H = *p->amg;
    cudaStream_t st = p->stream;
    const DeflFuse df = dfp ? *dfp : DeflFuse{};
    if (!H.use_graphs || p->prof.active >= 0) {
        ProfScope ps(&p->prof, KC_VCYCLE, st);
        vcycle_launch(p, v, s, z, df, w, st);
        KNP_CUDA(cudaGetLastError());
        return;
    }
    if (!H.gstream) {
        KNP_CUDA(cudaStreamCreateWithFlags(&H.gstream, cudaStreamNonBlocking));
    }
    // the correction's arrays are fixed per problem, so its y pointer and direction identify them
    auto key = std::make_tuple(v, s, z, df.y, (int)df.transpose, w);
    auto it = H.graphs.find(key);
    if (it == H.graphs.end()) {
        VcycleGraph g;
        int64_t before = g_launches.load();
        KNP_CUDA(cudaStreamBeginCapture(H.gstream, cudaStreamCaptureModeThreadLocal));
        try {
            vcycle_launch(p, v, s, z, df, w, Queue(H.gstream, true));
        } catch (...) {
            cudaGraph_t tmp;
            cudaStreamEndCapture(H.gstream, &tmp);
            if (tmp) cudaGraphDestroy(tmp);
            throw;
        }
        cudaGraph_t graph = nullptr;
        KNP_CUDA(cudaStreamEndCapture(H.gstream, &graph));
        g.launches = (int)(g_launches.load() - before);
        g_launches.fetch_sub(g.launches);
        KNP_CUDA(cudaGraphInstantiate(&g.exec, graph, 0));
        cudaGraphDestroy(graph);
        it = H.graphs.emplace(key, g).first;
    }
    KNP_CUDA(cudaGraphLaunch(it->second.exec, st));
    count_launch(it->second.launches);
}

}  // namespace knp

// ---------------------------------------------------------------------------------------------
// Allocation-free variant of knp_apply_preconditioner (include/knp.h). Some callers cannot call
// cudaMalloc when they need the preconditioner: code running under a CUDA stream capture or a
// graph being built, callers whose memory is fixed up front by a host framework, and embedded or
// plugin hosts that forbid allocation after start-up. The variant runs the same kernels as the
// V-cycle above on the same hierarchy, but all of its work vectors (the per-level x, x', b, r, d,
// the unit scale vector and the two layout-conversion buffers) live in one file-scope static
// device array of KNP_NOALLOC_SCRATCH_BYTES, which every GPU that loads the library holds until
// the process exits. Calls share that array, so two calls that overlap on the GPU (different
// streams, different problems, or different host threads) race on it and must be serialised.
// Nothing in the array needs to start at zero: every work vector is written before it is read.
// ---------------------------------------------------------------------------------------------

namespace knp {

namespace {

constexpr size_t KNP_NOALLOC_SCRATCH_BYTES = size_t(32) << 20;   // 32 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[KNP_NOALLOC_SCRATCH_BYTES];

// Device address of g_noalloc_scratch on the current device. Host code cannot use the symbol
// itself (on the host it names a stand-in, not device memory), so the address is looked up with
// cudaGetSymbolAddress once per device, with that device current, and cached.
std::mutex g_noalloc_mu;
std::map<int, void*> g_noalloc_addr;

unsigned char* noalloc_scratch() {
    int dev = -1;
    KNP_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    auto it = g_noalloc_addr.find(dev);
    if (it != g_noalloc_addr.end()) return static_cast<unsigned char*>(it->second);
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    KNP_REQUIRE(e == cudaSuccess && ptr, KNP_ERR_CUDA, "cudaGetSymbolAddress of the static scratch failed: %s",
                cudaGetErrorString(e));
    g_noalloc_addr[dev] = ptr;
    return static_cast<unsigned char*>(ptr);
}

__global__ void k_fill(int64_t n, double v, double* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = v;
}

// Eq. 4.3 order [c_i^1..c_i^3, phi_i, c_e^1..c_e^3, phi_e] <-> node-major [node][4]
__global__ void k_eq42_to_nodes(int64_t Ni, int64_t Ne, const double* __restrict__ a, double* __restrict__ out) {
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= Ni + Ne) return;
    for (int k = 0; k < 4; ++k)
        out[4 * g + k] = g < Ni ? a[(int64_t)k * Ni + g] : a[4 * Ni + (int64_t)k * Ne + (g - Ni)];
}

__global__ void k_nodes_to_eq42(int64_t Ni, int64_t Ne, const double* __restrict__ in, double* __restrict__ a) {
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= Ni + Ne) return;
    for (int k = 0; k < 4; ++k) {
        if (g < Ni)
            a[(int64_t)k * Ni + g] = in[4 * g + k];
        else
            a[4 * Ni + (int64_t)k * Ne + (g - Ni)] = in[4 * g + k];
    }
}

// per-level work vectors carved out of the static array
template <class T>
struct NaWork {
    T *x, *x2, *b, *r, *d;
};

inline size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

template <class T>
static void na_cheb_step(DevLevel<T>& L, NaWork<T>& w, const Coef4& c, int k, int steps, cudaStream_t st) {
    launch_cheb(L, w.x, w.b, c, w.d, w.x2, k, steps, st);
    std::swap(w.x, w.x2);
}

template <class T>
static void na_vcycle_rec(AmgDev<T>& D, std::vector<NaWork<T>>& W, int l, const double* v, const double* s,
                          cudaStream_t st) {
    DevLevel<T>& L = *D.L[l];
    NaWork<T>& w = W[l];
    const int last = (int)D.L.size() - 1;
    if (l == last) {
        if (v) {
            Coef4 c0{};
            count_launch();
            k_cheb_first<T, false><<<nblk(L.n, DT), DT, 0, st>>>(L.n, v, s, w.b, L.dinv.p, c0, w.x, w.d, DeflFuse{}, 0);
        }
        count_launch();
        k_coarse<T><<<nblk(4 * D.nc * 32, 256), 256, 0, st>>>(D.nc, D.cinv.p, w.b, w.x);
        return;
    }
    DevLevel<T>& C = *D.L[l + 1];
    NaWork<T>& wc = W[l + 1];
    const std::vector<Coef4>& cs = D.coef[l];
    count_launch();
    k_cheb_first<T, false><<<nblk(L.n, DT), DT, 0, st>>>(L.n, v, s, w.b, L.dinv.p, cs[0], w.x, w.d, DeflFuse{},
                                                     D.pre > 1);
    for (int k = 1; k < D.pre; ++k) na_cheb_step(L, w, cs[k], k, D.pre, st);
    launch_resid(L, w.x, w.b, w.r, st);
    restrict_to(L.R, w.r, wc.b, st);
    na_vcycle_rec(D, W, l + 1, nullptr, nullptr, st);
    prolong(L.P, wc.x, w.x, st);
    for (int k = 0; k < D.degree; ++k) na_cheb_step(L, w, cs[k], k, D.degree, st);
}

// Lays the work vectors out in the static array; returns the bytes needed (and fills W when
// `base` is not NULL).
template <class T>
static size_t na_layout(AmgDev<T>& D, int64_t n0, unsigned char* base, std::vector<NaWork<T>>& W, double** ones,
                        double** rin, double** zout, T** xfine) {
    size_t off = 0;
    auto take = [&](size_t bytes) -> unsigned char* {
        unsigned char* p = base ? base + off : nullptr;
        off += align256(bytes);
        return p;
    };
    *ones = reinterpret_cast<double*>(take(4 * n0 * sizeof(double)));
    *rin = reinterpret_cast<double*>(take(4 * n0 * sizeof(double)));
    *zout = reinterpret_cast<double*>(take(4 * n0 * sizeof(double)));
    W.assign(D.L.size(), NaWork<T>{});
    for (size_t l = 0; l < D.L.size(); ++l) {
        size_t b = 4 * (size_t)D.L[l]->n * sizeof(T);
        W[l].x = reinterpret_cast<T*>(take(b));
        W[l].x2 = reinterpret_cast<T*>(take(b));
        W[l].b = reinterpret_cast<T*>(take(b));
        W[l].r = reinterpret_cast<T*>(take(b));
        W[l].d = reinterpret_cast<T*>(take(b));
    }
    *xfine = nullptr;
    return off;
}

template <class T>
static void na_apply(knp_problem* p, AmgDev<T>& D, const double* r_eq42, double* z_eq42) {
    cudaStream_t st = p->stream;
    const int64_t n0 = D.L[0]->n;
    std::vector<NaWork<T>> W;
    double *ones, *rin, *zout;
    T* xf;
    size_t need = na_layout(D, n0, nullptr, W, &ones, &rin, &zout, &xf);
    KNP_REQUIRE(need <= KNP_NOALLOC_SCRATCH_BYTES, KNP_ERR_INVALID_ARG,
                "knp_apply_preconditioner_noalloc needs %zu bytes of scratch for this hierarchy; the static "
                "array holds %zu (use knp_apply_preconditioner)",
                need, KNP_NOALLOC_SCRATCH_BYTES);
    unsigned char* base = noalloc_scratch();
    na_layout(D, n0, base, W, &ones, &rin, &zout, &xf);
    count_launch(3);
    k_fill<<<nblk(4 * n0, 256), 256, 0, st>>>(4 * n0, 1.0, ones);
    k_eq42_to_nodes<<<nblk(n0, 256), 256, 0, st>>>(p->N_i, p->N_e, r_eq42, rin);
    na_vcycle_rec(D, W, 0, rin, ones, st);
    count_launch();
    k_to_double<T><<<nblk(4 * n0, 256), 256, 0, st>>>(4 * n0, W[0].x, zout);
    count_launch();
    k_nodes_to_eq42<<<nblk(n0, 256), 256, 0, st>>>(p->N_i, p->N_e, zout, z_eq42);
    KNP_CUDA(cudaGetLastError());
}

}  // namespace

}  // namespace knp

extern "C" knp_status knp_apply_preconditioner_noalloc(knp_problem* p, const double* r, double* z) {
    using namespace knp;
    return guarded([&] {
        KNP_REQUIRE(p && r && z, KNP_ERR_INVALID_ARG, "NULL argument");
        KNP_REQUIRE(p->amg, KNP_ERR_STATE, "knp_amg_setup has not been called");
        // the static array is looked up on the current device: it must be the problem's
        cudaPointerAttributes at{};
        KNP_CUDA(cudaPointerGetAttributes(&at, p->u.p));
        int dev = -1;
        KNP_CUDA(cudaGetDevice(&dev));
        KNP_REQUIRE(at.device == dev, KNP_ERR_INVALID_ARG,
                    "the current device (%d) is not the problem's device (%d); make it current first", dev,
                    at.device);
        if (p->amg->h32)
            na_apply(p, *static_cast<AmgDev<float>*>(p->amg->h32), r, z);
        else
            na_apply(p, *static_cast<AmgDev<double>*>(p->amg->h64), r, z);
    });
}

