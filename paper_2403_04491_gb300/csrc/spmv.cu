// y = A_{n-1} x on the node-block structure of Section 4.1.
//
// Per directed same-region entry (j, l) the operator stores five numbers: the mass
// m_jl and stiffness a_jl (static) and e^k_jl = tau~_r^k A_r^{k,n-1}_jl + [C_r^k M_{r,Gamma}]_jl
// (per step). The 4x4 node block of A_r^n is then
//     c^k row:  (m + tau_r^k a) on c^k,   e^k on phi_r
//     phi row:  z_k tau_r^k a on c^k,     sum_k z_k e^k on phi_r
// because sum_k z_k C_r^k = C_m/F (sum_k alpha_r^k = 1). Cross-region membrane entries
// (B_rq) carry -[C_r^k M_{rq,Gamma}] in the same e^k slot with m = a = 0.
//
// GB300 issues FP64 at 1/64 of its FP32 rate, so the forward product is bound by FP64 FMAs, not
// by bytes. It therefore reads the static per-ion sums g^k = m + tau_r^k a (folded once at
// problem creation) and, for the potential row, a per-node w = sum_k z_k tau_r^k x^k made by a
// small pass over the nodes first (or by
// the V-cycle's last kernel, when x is its result):
//     c^k row:  sum g^k x^k + sum e^k phi,     phi row:  sum a w + sum_k z_k (sum e^k phi),
// seven FMAs per stored entry (g^k x^k, e^k phi, a w) for 60 bytes, where m, a with the
// per-row tau take nine for 44 bytes. The transposed product keeps the m, a form.
// One, four or eight lanes per row (lanes.h); the sliced-ELL layout makes the value loads of a warp
// contiguous.
//
// Point pin (Remark 4.1): the stored values keep the phi_e column of the pinned node (so the
// same-region values stay symmetric and serve the transpose too); both kernels treat that
// column as zero and give the pinned phi_e row the identity.
#include <algorithm>

#include "lanes.h"
#include "launch.h"
#include "problem.h"

namespace knp {

namespace {

struct OpArgs {
    int64_t n, N_i, n_entries;
    int32_t pin;
    const int64_t* slice_ptr;
    const int32_t* col;
    const double* m;
    const double* a;
    const double* e;
    const double* g;        // [3][n_entries] g^k = m + tau_r^k a of the entry's region (static)
    const double* w;        // [n] sum_k z_k tau_r^k x^k per node (made by k_op_w)
    const int32_t* xptr;
    const int32_t* xcol;
    const double* xe;
    int64_t n_cross;
    const int32_t* xtptr;   // transposed cross-region entries: row -> (source row, value index)
    const int32_t* xtrow;
    const int32_t* xtidx;
    double tau[2][KI];
    double z[KI];
};

// w[c] = sum_k z_k tau_r^k x^k[c], r the region of node c
__global__ void k_op_w(OpArgs A, const double* x, double* __restrict__ w) {
    chain_wait();
    int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= A.n) return;
    const int reg = c < A.N_i ? 0 : 1;
    const double2* xp = reinterpret_cast<const double2*>(x + 4 * c);
    const double2 x01 = xp[0], x23 = xp[1];
    w[c] = A.z[0] * A.tau[reg][0] * x01.x + A.z[1] * A.tau[reg][1] * x01.y + A.z[2] * A.tau[reg][2] * x23.x;
}

// y = rowscale .* (b - A x)  (b, rowscale optional) on the fields of row r that a lane holds in out
template <int F>
__device__ __forceinline__ void op_store(int64_t k, const double* out, double* __restrict__ y,
                                         const double* __restrict__ rowscale, const double* b) {
    double o[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
        o[f] = out[f];
        if (b) o[f] = b[k + f] - o[f];
        if (rowscale) o[f] *= rowscale[k + f];
    }
    if constexpr (F == 4) {
        double2* yp = reinterpret_cast<double2*>(y + k);
        yp[0] = make_double2(o[0], o[1]);
        yp[1] = make_double2(o[2], o[3]);
    } else {
#pragma unroll
        for (int f = 0; f < F; ++f) y[k + f] = o[f];
    }
}

// y = rowscale .* (b - A x)  (b, rowscale optional), L lanes per row (lanes.h). One and four lanes per
// row read w = k_op_w(x); with eight the kernel is bound by its chain of loads, so it forms w from
// the x it gathers anyway (three FMAs per entry). Read by four lanes, 117,504 unknowns in 3D 9.75 -> 9.53 ms
// for three steps, P2 20^3 26.3 -> 24.8 for two; by eight, the Kir problem on 97x75 6.77 -> 6.90. The loads
// of OP_BATCH entries are issued together.
template <int L>
constexpr int OP_BATCH = L == 1 ? 1 : 3;
template <int L>
__global__ void __launch_bounds__(128) k_op_apply(OpArgs A, const double* x, double* __restrict__ y,
                                                  const double* __restrict__ rowscale, const double* b) {
    constexpr int F = LANE_FIELDS<L>, U = OP_BATCH<L>;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t r = gid / L;
    const int t = (int)(gid % L);
    if (L == 1 && r >= A.n) return;   // with more lanes, all of a warp take part in the shuffles
    const int64_t row = r < A.n ? r : A.n - 1;
    const int reg = row < A.N_i ? 0 : 1;
    const int64_t s = row / SELL_C;
    const int64_t base = A.slice_ptr[s] + row % SELL_C;
    const int w = (int)((A.slice_ptr[s + 1] - A.slice_ptr[s]) / SELL_C);
    const int64_t ne = A.n_entries;
    const int32_t* cp = A.col + base;
    const double *g0 = A.g + base, *e0 = A.e + base, *ap = A.a + base;
    double ag[KI] = {0, 0, 0}, ae[KI] = {0, 0, 0}, aw = 0.0;
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = t + u * L < w ? cp[(t + u * L) * SELL_C] : 0;
    chain_wait();
    for (int k = t; k < w; k += U * L) {
        double2 x01[U], x23[U];
        double gv[U][KI], ev[U][KI], av[U], wv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w) {
                const int q = (k + u * L) * SELL_C;
                const double2* xp = reinterpret_cast<const double2*>(x + 4 * (int64_t)c[u]);
                x01[u] = xp[0];
                x23[u] = xp[1];
                if (L <= 4) wv[u] = A.w[c[u]];
#pragma unroll
                for (int i = 0; i < KI; ++i) {
                    gv[u][i] = g0[i * ne + q];
                    ev[u][i] = e0[i * ne + q];
                }
                av[u] = ap[q];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w) {
                const double phi = (c[u] == A.pin) ? 0.0 : x23[u].y;
                if (L > 4)
                    wv[u] = A.z[0] * A.tau[reg][0] * x01[u].x + A.z[1] * A.tau[reg][1] * x01[u].y +
                            A.z[2] * A.tau[reg][2] * x23[u].x;
                ag[0] += gv[u][0] * x01[u].x;
                ag[1] += gv[u][1] * x01[u].y;
                ag[2] += gv[u][2] * x23[u].x;
                aw += av[u] * wv[u];
#pragma unroll
                for (int i = 0; i < KI; ++i) ae[i] += ev[u][i] * phi;
            }
            const int q = k + (U + u) * L;
            c[u] = q < w ? cp[q * SELL_C] : 0;
        }
    }
    for (int u = A.xptr[row] + t; u < A.xptr[row + 1]; u += L) {
        int64_t cc = A.xcol[u];
        double phi = (cc == A.pin) ? 0.0 : x[4 * cc + 3];
        for (int k = 0; k < KI; ++k) ae[k] += A.xe[k * A.n_cross + u] * phi;
    }
    double out[4], mine[F];
    out[3] = aw;
    for (int k = 0; k < KI; ++k) {
        out[k] = ag[k] + ae[k];
        out[3] += A.z[k] * ae[k];
    }
    lane_reduce4<double, L>(out, t, mine);
    if (r >= A.n || t >= 4) return;
    const int f0 = lane_field<L>(t);
    if (r == A.pin && f0 + F == 4) mine[F - 1] = x[4 * r + 3];
    op_store<F>(4 * r + f0, mine, y, rowscale, b);
}

// g^k = m + tau_r^k a per stored entry (padding included, where m = a = 0)
__global__ void k_fold_g(int64_t n, int64_t N_i, int64_t ne, const int64_t* __restrict__ slice_ptr,
                         const double* __restrict__ m, const double* __restrict__ a, double ti0, double ti1, double ti2,
                         double te0, double te1, double te2, double* __restrict__ g) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    const bool in = r < N_i;
    const double t[3] = {in ? ti0 : te0, in ? ti1 : te1, in ? ti2 : te2};
    const int64_t s = r / SELL_C, base = slice_ptr[s] + r % SELL_C;
    const int64_t w = (slice_ptr[s + 1] - slice_ptr[s]) / SELL_C;
    for (int64_t k = 0; k < w; ++k) {
        const int64_t pos = base + k * SELL_C;
        for (int q = 0; q < KI; ++q) g[q * ne + pos] = m[pos] + t[q] * a[pos];
    }
}

// y = rowscale .* (b - A^T x): the transposed node block of entry (j, l) is
//     c^k row:  (m + tau^k a) x^k_j + z_k tau^k a x^phi_j,   phi row:  sum_k e^k (x^k_j + z_k x^phi_j)
// with m, a, e symmetric on same-region entries; the cross-region part uses the transposed list.
template <int L>
__global__ void __launch_bounds__(128) k_op_apply_t(OpArgs A, const double* x, double* __restrict__ y,
                                                    const double* __restrict__ rowscale, const double* b) {
    constexpr int F = LANE_FIELDS<L>, U = OP_BATCH<L>;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t r = gid / L;
    const int t = (int)(gid % L);
    if (L == 1 && r >= A.n) return;
    const int64_t row = r < A.n ? r : A.n - 1;
    const int reg = row < A.N_i ? 0 : 1;
    const int64_t s = row / SELL_C;
    const int64_t base = A.slice_ptr[s] + row % SELL_C;
    const int w = (int)((A.slice_ptr[s + 1] - A.slice_ptr[s]) / SELL_C);
    const int64_t ne = A.n_entries;
    const int32_t* cp = A.col + base;
    const double *mp = A.m + base, *e0 = A.e + base, *ap0 = A.a + base;
    double am[KI] = {0, 0, 0}, aa[KI] = {0, 0, 0}, ap = 0.0, ae = 0.0;
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = t + u * L < w ? cp[(t + u * L) * SELL_C] : 0;
    chain_wait();
    for (int k = t; k < w; k += U * L) {
        double2 x01[U], x23[U];
        double ev[U][KI], mv[U], av[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w) {
                const int q = (k + u * L) * SELL_C;
                const double2* xp = reinterpret_cast<const double2*>(x + 4 * (int64_t)c[u]);
                x01[u] = xp[0];
                x23[u] = xp[1];
#pragma unroll
                for (int i = 0; i < KI; ++i) ev[u][i] = e0[i * ne + q];
                mv[u] = mp[q];
                av[u] = ap0[q];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k + u * L < w) {
                const double xc[KI] = {x01[u].x, x01[u].y, x23[u].x};
                const double phi = (c[u] == A.pin) ? 0.0 : x23[u].y;
#pragma unroll
                for (int i = 0; i < KI; ++i) {
                    am[i] += mv[u] * xc[i];
                    aa[i] += av[u] * xc[i];
                    ae += ev[u][i] * (xc[i] + A.z[i] * phi);
                }
                ap += av[u] * phi;
            }
            const int q = k + (U + u) * L;
            c[u] = q < w ? cp[q * SELL_C] : 0;
        }
    }
    for (int u = A.xtptr[row] + t; u < A.xtptr[row + 1]; u += L) {
        int64_t j = A.xtrow[u];
        int64_t idx = A.xtidx[u];
        double phi = (j == A.pin) ? 0.0 : x[4 * j + 3];
        for (int q = 0; q < KI; ++q) ae += A.xe[q * A.n_cross + idx] * (x[4 * j + q] + A.z[q] * phi);
    }
    double out[4], mine[F];
    for (int q = 0; q < KI; ++q) out[q] = am[q] + A.tau[reg][q] * (aa[q] + A.z[q] * ap);
    out[3] = ae;
    lane_reduce4<double, L>(out, t, mine);
    if (r >= A.n || t >= 4) return;
    const int f0 = lane_field<L>(t);
    if (r == A.pin && f0 + F == 4) mine[F - 1] = x[4 * r + 3];
    op_store<F>(4 * r + f0, mine, y, rowscale, b);
}

}  // namespace

static int op_lanes(const knp_problem* p) {
    return row_lanes(p->n_nodes, (double)p->sell.n_entries / (double)std::max<int64_t>(p->n_nodes, 1));
}

bool op_reads_w(const knp_problem* p) { return op_lanes(p) <= 4; }

void op_apply(knp_problem* p, const double* x, double* y, const double* rowscale, const double* b, bool transpose,
              Queue q, bool w_ready) {
    if (q.st == kProblemStream) q.st = p->stream;
    OpArgs A;
    A.n = p->n_nodes;
    A.N_i = p->N_i;
    A.n_entries = p->sell.n_entries;
    A.pin = p->pin;
    A.slice_ptr = p->sell.slice_ptr.p;
    A.col = p->sell.col.p;
    A.m = p->sell_m.p;
    A.a = p->sell_a.p;
    A.e = p->sell_e.p;
    A.g = p->sell_g.p;
    A.w = p->op_w.p;
    A.xptr = p->xptr.p;
    A.xcol = p->xcol.p;
    A.xe = p->xe.p;
    A.n_cross = (int64_t)p->h_xcol.size();
    A.xtptr = p->xtptr.p;
    A.xtrow = p->xtrow.p;
    A.xtidx = p->xtidx.p;
    for (int r = 0; r < 2; ++r)
        for (int k = 0; k < KI; ++k) A.tau[r][k] = p->sp.reg[r].tau[k];
    for (int k = 0; k < KI; ++k) A.z[k] = p->sp.z[k];
    const int lanes = op_lanes(p);
    const unsigned blocks = (unsigned)((A.n * lanes + 127) / 128);
    ProfScope ps(&p->prof, KC_SPMV, q.st);
    count_launch();
    if (transpose) {
        if (lanes == 1)
            launch(k_op_apply_t<1>, blocks, 128, q, A, x, y, rowscale, b);
        else if (lanes == 4)
            launch(k_op_apply_t<4>, blocks, 128, q, A, x, y, rowscale, b);
        else
            launch(k_op_apply_t<8>, blocks, 128, q, A, x, y, rowscale, b);
        KNP_CUDA(cudaGetLastError());
        return;
    }
    if (op_reads_w(p) && !w_ready) {
        count_launch();
        launch(k_op_w, (A.n + 255) / 256, 256, q, A, x, p->op_w.p);
    }
    if (lanes == 1) {
        launch(k_op_apply<1>, blocks, 128, q, A, x, y, rowscale, b);
    } else if (lanes == 4) {
        launch(k_op_apply<4>, blocks, 128, q, A, x, y, rowscale, b);
    } else {
        launch(k_op_apply<8>, blocks, 128, q, A, x, y, rowscale, b);
    }
    KNP_CUDA(cudaGetLastError());
}

void op_prepare(knp_problem* p, cudaStream_t st) {
    const int64_t n = p->n_nodes, ne = p->sell.n_entries;
    p->sell_g.alloc(std::max<int64_t>(1, 3 * ne));
    p->op_w.alloc(std::max<int64_t>(1, n));
    const RegionCoef& ri = p->sp.reg[0];
    const RegionCoef& re = p->sp.reg[1];
    count_launch();
    k_fold_g<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(n, p->N_i, ne, p->sell.slice_ptr.p, p->sell_m.p, p->sell_a.p,
                                                          ri.tau[0], ri.tau[1], ri.tau[2], re.tau[0], re.tau[1],
                                                          re.tau[2], p->sell_g.p);
    KNP_CUDA(cudaGetLastError());
}

}  // namespace knp
