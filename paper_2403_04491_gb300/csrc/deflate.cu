// Coarse correction of the potentials' near-null modes, wrapped around P_0^{-1} (Section 4.2).
//
// The potential blocks of P_0 are nearly singular: the intracellular potential of each cell is held
// only by the membrane capacitance (C_m/F M_Gamma, small against the stiffness of the cell's
// interior) and the extracellular potential only by the point pin of Remark 4.1. One V-cycle
// applies P_0^{-1} to these modes correctly, but a residual component along them is amplified by
// about 1/lambda_min. The paper's left-preconditioned GMRES minimises the preconditioned residual
// and so works on exactly that amplified quantity; the right-preconditioned FGMRES used here
// minimises the residual, which barely sees these modes, while its stopping test measures the
// preconditioned residual: without help the test stagnates far above its threshold (on the paper's
// 1 um Model A as well as at 100 um).
//
// The remedy is a two-level preconditioner with the coarse space Z = the per-cell constants of
// phi_i and the constant of phi_e (the pinned node left out), on the true operator:
//     E = Z^T A Z,   y = E^{-1} Z^T r,   M_D^{-1} r = P_0^{-1} (r - A Z y) + Z y.
// The V-cycle then sees a residual orthogonal to Z (nothing left to amplify) and Z y is the exact
// correction of those modes. FGMRES tolerates any preconditioner, so the iterate's accuracy is
// still set by the stopping test alone. The adjoint's A^T solve uses the same coarse space with
// Z^T A^T Z = E^T.
//
// Costs. A applied to a piecewise-constant potential is nonzero only through the membrane and
// pin terms: the same-region row sums of e^k (and of a) vanish except at the active rows, the membrane
// nodes and the pinned node with its neighbours, since every assembled diagonal is minus its row's sum.
// So A Z y is nonzero at the active rows alone (a few percent of the nodes), and there it is a fixed
// combination of two constants, the node's own group's and the one on the membrane's other side; the
// eight coefficients of an active row are formed once per step. E is an arrowhead matrix
// (cells couple only to the extracellular space) solved by its Schur complement on the device, and each
// application adds a gather and a small solve; the right-hand-side pass and the update run inside the
// V-cycle's first and last kernels (CG(P_0) keeps them as separate passes).
// Sums are taken in a fixed order (no atomics), so the result is reproducible bit for bit. They are
// split into chunks of GATHER_NODES nodes, also within a cell: one block per cell took 37 us per
// application and 546 us per step for the one cell of the 64^3 workload.
#include <algorithm>
#include <map>
#include <memory>
#include <utility>
#include <vector>

#include "deflate.h"
#include "deflate_input.h"
#include "problem.h"
#include "vcycle.h"

namespace knp {

namespace {

constexpr int GATHER_NODES = 1024;   // nodes per block of the gather
constexpr int EXT_BLOCKS = 304;      // most partial sums over the extracellular nodes

// Coefficients of active row i, formed once per step: (A Z y)_f = C[f] y_own + C[4 + f] y_cross for its
// four fields f, and (A^T Z y)_f likewise with CT. A Z y: the row's same-region phi columns other than
// the pin hold its own group's constant (sums of e^k), its cross-region entries that of the one group on
// the membrane's other side (a membrane node touches one cell only, so all its entries share it; xgrp);
// the potential row is sum_k z_k of the concentration rows' terms. A^T Z y: tau_r^k z_k times the row
// sum of a on the concentrations, sum_k z_k e^k and, through the transposed list, sum_k z_k xe^k on the
// potential. The pinned potential row (the identity) gives 0.
__global__ void k_defl_coefs(int64_t na, int64_t N_i, int32_t pin, const int32_t* __restrict__ rows,
                             const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ col,
                             const double* __restrict__ e, int64_t ne, const double* __restrict__ a,
                             const int32_t* __restrict__ xptr, const int32_t* __restrict__ xcol,
                             const int32_t* __restrict__ xtptr, const int32_t* __restrict__ xtrow,
                             const int32_t* __restrict__ xtidx, const double* __restrict__ xe, int64_t n_cross,
                             double z0, double z1, double z2, RegionCoef ri, RegionCoef re, double* __restrict__ C,
                             double* __restrict__ CT) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= na) return;
    const int64_t r = rows[i];
    const int64_t s = r / SELL_C, base = slice_ptr[s] + r % SELL_C;
    const int w = (int)((slice_ptr[s + 1] - slice_ptr[s]) / SELL_C);
    const double z[KI] = {z0, z1, z2};
    double own[KI] = {0, 0, 0}, cross[KI] = {0, 0, 0}, sa = 0.0, ct = 0.0;
    for (int k = 0; k < w; ++k) {
        const int64_t pos = base + k * SELL_C;
        if (col[pos] == pin) continue;
        for (int q = 0; q < KI; ++q) own[q] += e[q * ne + pos];
        sa += a[pos];
    }
    for (int t = xptr[r]; t < xptr[r + 1]; ++t) {
        if (xcol[t] == pin) continue;
        for (int q = 0; q < KI; ++q) cross[q] += xe[q * n_cross + t];
    }
    for (int t = xtptr[r]; t < xtptr[r + 1]; ++t) {
        if (xtrow[t] == pin) continue;
        const int64_t idx = xtidx[t];
        for (int q = 0; q < KI; ++q) ct += z[q] * xe[q * n_cross + idx];
    }
    const bool in = r < N_i, free = r != pin;
    double* c = C + 8 * i;
    double* t = CT + 8 * i;
    double po = 0.0, pc = 0.0;
    for (int q = 0; q < KI; ++q) {
        c[q] = own[q];
        c[4 + q] = cross[q];
        po += z[q] * own[q];
        pc += z[q] * cross[q];
        t[q] = (in ? ri.tau[q] : re.tau[q]) * z[q] * sa;
        t[4 + q] = 0.0;
    }
    c[3] = t[3] = free ? po : 0.0;
    c[7] = free ? pc : 0.0;
    t[7] = free ? ct : 0.0;
}

// Chunk b of a cell group's active rows (one block): its share of E_jj, E_je and E_ej of E = Z^T A Z,
// the sums of the potential rows' coefficients of A Z and (for E_ej) of A^T Z. Blocks from nchunks on:
// one chunk each of the extracellular active rows' share of E_ee.
__global__ void __launch_bounds__(DT) k_defl_E(int nchunks, const int64_t* __restrict__ cbeg,
                                               const int32_t* __restrict__ aidx, int64_t ext0, int64_t na,
                                               const double* __restrict__ C, const double* __restrict__ CT,
                                               double* __restrict__ part) {
    __shared__ double sh[DT / 32];
    const int b = blockIdx.x;
    double djj = 0.0, dje = 0.0, dej = 0.0;
    if (b < nchunks) {
        const int64_t q = cbeg[b] + threadIdx.x;
        if (q < cbeg[b + 1]) {
            const int64_t i = aidx[q];
            djj = C[8 * i + 3];
            dje = C[8 * i + 7];
            dej = CT[8 * i + 7];
        }
    } else {
        const int64_t i = ext0 + (b - nchunks) * (int64_t)DT + threadIdx.x;
        if (i < na) djj = C[8 * i + 3];
    }
    double a = block_sum(djj, sh);
    if (threadIdx.x == 0) part[3 * b] = a;
    a = block_sum(dje, sh);
    if (threadIdx.x == 0) part[3 * b + 1] = a;
    a = block_sum(dej, sh);
    if (threadIdx.x == 0) part[3 * b + 2] = a;
}

// 1 / E_jj, E_je, E_ej of each group from its chunks' shares; E_ee and one over the Schur complement
// S_e = E_ee - sum_j E_ej E_je / E_jj (one block)
__global__ void __launch_bounds__(DT) k_defl_schur(int nc, int nchunks, int next, const int32_t* __restrict__ cchunk,
                                                   const double* __restrict__ part, double* __restrict__ iEjj,
                                                   double* __restrict__ Eje, double* __restrict__ Eej,
                                                   double* __restrict__ Ee) {
    __shared__ double sh[DT / 32];
    double a = 0.0, b = 0.0;
    for (int q = threadIdx.x; q < next; q += blockDim.x) a += part[3 * (int64_t)(nchunks + q)];
    for (int j = threadIdx.x; j < nc; j += blockDim.x) {
        double jj = 0.0, je = 0.0, ej = 0.0;
        for (int64_t q = cchunk[j]; q < cchunk[j + 1]; ++q) {
            jj += part[3 * q];
            je += part[3 * q + 1];
            ej += part[3 * q + 2];
        }
        iEjj[j] = 1.0 / jj;
        Eje[j] = je;
        Eej[j] = ej;
        b += ej * je / jj;
    }
    const double eee = block_sum(a, sh);
    const double red = block_sum(b, sh);
    if (threadIdx.x == 0) {
        Ee[0] = eee;
        Ee[1] = 1.0 / (eee - red);
    }
}

// partial sums of g = Z^T r with r = s .* v
__global__ void __launch_bounds__(DT) k_defl_gather(GatherArgs a, const double* v, const double* __restrict__ s) {
    __shared__ double sh[DT / 32];
    chain_wait();
    const double t = block_sum(gather_share(a, blockIdx.x, [&](int64_t k) { return s[k] * v[k]; }), sh);
    if (threadIdx.x == 0) a.part[blockIdx.x] = t;
}

// y = E^{-1} g (one block)
__global__ void __launch_bounds__(DT) k_defl_solve(CoarseSolve e, double* y) {
    chain_wait();
    coarse_solve(e, y);
}

// t = s .* v - A Z y (or - A^T Z y), for CG(P_0)
__global__ void k_defl_rhs(int64_t n, const double* __restrict__ v, const double* __restrict__ s, DeflFuse df,
                           double* __restrict__ t) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    double o[4];
    defl_input(r, v, s, df, df.y, o);
    for (int q = 0; q < 4; ++q) t[4 * r + q] = o[q];
}

// z += Z y: the potential of every node of a group takes its group's constant
__global__ void k_defl_add(int64_t n, int64_t N_i, int32_t pin, const int32_t* __restrict__ rgrp,
                           const double* __restrict__ y, int32_t ext_group, double* __restrict__ z) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n || r == pin) return;
    z[4 * r + 3] += y[r < N_i ? rgrp[r] : ext_group];
}

__global__ void k_fill_ones(int64_t n, double* __restrict__ v) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) v[i] = 1.0;
}

inline unsigned nbk(int64_t n, int t) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

}  // namespace

struct Deflation {
    int nc = 0;                       // cell groups (cells with at least one intracellular node)
    int64_t na = 0, na_i = 0;         // active rows, and the intracellular ones (first) among them
    int gchunks = 0, echunks = 0;     // chunks of the cells' nodes (gather) and active rows (E)
    int gext = 0, eext = 0;           // blocks of the extracellular sums of the two
    DArray<int64_t> gbeg, ebeg;       // chunk -> its first entry of cnodes / aidx
    DArray<int32_t> gcell, ecell;     // group -> its first chunk
    DArray<int32_t> cnodes;           // intracellular nodes by group (increasing)
    DArray<int32_t> aidx;             // intracellular active rows by group, as indices into rows
    DArray<int32_t> rows;             // active rows (increasing)
    DArray<int32_t> act;              // node -> its index in rows, -1 if not active
    DArray<int32_t> rgrp;             // intracellular node -> its group
    DArray<int32_t> xgrp;             // active row -> group on the membrane's other side
    DArray<double> C, CT;             // [na][8] coefficients of A Z y and A^T Z y (per step)
    DArray<double> iEjj, Eje, Eej;    // the arrowhead E (per step): 1 / E_jj, E_je, E_ej
    DArray<double> Ee;                // {E_ee, 1 / Schur complement}
    DArray<double> y, gpart, epart;
    DArray<double> t, ones;           // CG(P_0)'s separate passes, on first use
    int64_t built_for = -1;           // assembly whose operator E was formed from
};

void deflation_free(Deflation* d) { delete d; }

// Splits the lists of each group (gptr: group -> first entry) into chunks of at most `most` entries
static void make_chunks(const std::vector<int64_t>& gptr, int64_t most, std::vector<int64_t>& beg,
                        std::vector<int32_t>& first) {
    beg.clear();
    first.assign(1, 0);
    for (size_t j = 0; j + 1 < gptr.size(); ++j) {
        for (int64_t q = gptr[j]; q < gptr[j + 1]; q += most) beg.push_back(q);
        first.push_back((int32_t)beg.size());
    }
    beg.push_back(gptr.back());
}

static Deflation& deflation_setup(knp_problem* p) {
    if (p->defl) return *p->defl;
    auto d = std::make_unique<Deflation>();   // the problem's once it is whole: an allocation may fail
    cudaStream_t st = p->stream;
    const knp_mesh& m = *p->mesh;
    const std::vector<int32_t>& cell = p->degree == 2 ? p2_nodes(m).node_cell_i : m.node_cell_i;
    KNP_REQUIRE((int64_t)cell.size() == p->N_i, KNP_ERR_STATE, "cell map does not match the intracellular nodes");
    const int64_t n = p->n_nodes;
    std::map<int32_t, int> gid;
    for (int32_t c : cell) gid.emplace(c, 0);
    int k = 0;
    for (auto& kv : gid) kv.second = k++;
    d->nc = k;
    std::vector<int32_t> rg(std::max<int64_t>(p->N_i, 1), 0);
    for (int64_t r = 0; r < p->N_i; ++r) rg[r] = gid[cell[r]];
    // active rows: membrane nodes (they have cross-region entries) and the rows with the pin's column,
    // which by the pattern's symmetry are the columns of the pin's row
    std::vector<uint8_t> on(n, 0);
    for (int64_t r = 0; r < n; ++r) on[r] = p->h_xptr[r + 1] > p->h_xptr[r];
    {
        const SellPattern& S = p->sell;
        const int64_t s = p->pin / SELL_C;
        for (int64_t q = S.h_slice_ptr[s] + p->pin % SELL_C; q < S.h_slice_ptr[s + 1]; q += SELL_C) on[S.h_col[q]] = 1;
    }
    std::vector<int32_t> rows, act(n, -1);
    for (int64_t r = 0; r < n; ++r)
        if (on[r]) {
            act[r] = (int32_t)rows.size();
            rows.push_back((int32_t)r);
            d->na_i += r < p->N_i;
        }
    d->na = (int64_t)rows.size();
    // entries [0, count) of a list (list[q]: intracellular node of entry q) by group, stably
    auto by_group = [&](int64_t count, auto node_of, std::vector<int64_t>& gptr, std::vector<int32_t>& out) {
        gptr.assign(d->nc + 1, 0);
        for (int64_t q = 0; q < count; ++q) gptr[rg[node_of(q)] + 1]++;
        for (int j = 0; j < d->nc; ++j) gptr[j + 1] += gptr[j];
        out.assign(std::max<int64_t>(count, 1), 0);
        std::vector<int64_t> fill(gptr.begin(), gptr.end() - 1);
        for (int64_t q = 0; q < count; ++q) out[fill[rg[node_of(q)]]++] = (int32_t)q;
    };
    std::vector<int64_t> gptr, beg;
    std::vector<int32_t> list, first;
    by_group(p->N_i, [](int64_t q) { return q; }, gptr, list);
    make_chunks(gptr, GATHER_NODES, beg, first);
    d->gchunks = (int)beg.size() - 1;
    d->gext = (int)std::min<int64_t>(EXT_BLOCKS, std::max<int64_t>(1, (p->N_e + GATHER_NODES - 1) / GATHER_NODES));
    d->cnodes.upload(list, st);
    d->gbeg.upload(beg, st);
    d->gcell.upload(first, st);
    by_group(d->na_i, [&](int64_t q) { return (int64_t)rows[q]; }, gptr, list);
    make_chunks(gptr, DT, beg, first);
    d->echunks = (int)beg.size() - 1;
    d->eext = (int)std::max<int64_t>(1, (d->na - d->na_i + DT - 1) / DT);
    d->aidx.upload(list, st);
    d->ebeg.upload(beg, st);
    d->ecell.upload(first, st);
    const int32_t ext = d->nc;
    std::vector<int32_t> xgrp(d->na, 0);   // rows without a usable cross entry have zero coefficients
    for (int64_t i = 0; i < d->na; ++i) {
        int32_t group = -1;
        for (int32_t t = p->h_xptr[rows[i]]; t < p->h_xptr[rows[i] + 1]; ++t) {
            const int32_t c = p->h_xcol[t];
            if (c == p->pin) continue;
            const int32_t gc = c < p->N_i ? rg[c] : ext;
            KNP_REQUIRE(group < 0 || group == gc, KNP_ERR_INVALID_MESH, "a membrane node touches two cells");
            group = gc;
        }
        if (group >= 0) xgrp[i] = group;
    }
    d->rows.upload(rows, st);
    d->act.upload(act, st);
    d->rgrp.upload(rg, st);
    d->xgrp.upload(xgrp, st);
    d->C.alloc(8 * d->na);
    d->CT.alloc(8 * d->na);
    for (DArray<double>* a : {&d->iEjj, &d->Eje, &d->Eej}) a->alloc(std::max(d->nc, 1));
    d->Ee.alloc(2);
    d->y.alloc(d->nc + 1);
    d->gpart.alloc(d->gchunks + d->gext);
    d->epart.alloc(3 * (d->echunks + d->eext));
    KNP_CUDA(cudaGetLastError());
    // the host tables above go out of scope here
    KNP_CUDA(cudaStreamSynchronize(st));
    p->defl = d.release();
    return *p->defl;
}

void deflation_prepare(knp_problem* p) {
    Deflation& d = deflation_setup(p);
    if (d.built_for == p->assembly_id) return;
    cudaStream_t st = p->stream;
    const int64_t nx = (int64_t)p->h_xcol.size();
    const double* z = p->sp.z;
    count_launch(3);
    k_defl_coefs<<<nbk(d.na, 64), 64, 0, st>>>(d.na, p->N_i, p->pin, d.rows.p, p->sell.slice_ptr.p, p->sell.col.p,
                                               p->sell_e.p, p->sell.n_entries, p->sell_a.p, p->xptr.p, p->xcol.p,
                                               p->xtptr.p, p->xtrow.p, p->xtidx.p, p->xe.p, nx, z[0], z[1], z[2],
                                               p->sp.reg[0], p->sp.reg[1], d.C.p, d.CT.p);
    k_defl_E<<<d.echunks + d.eext, DT, 0, st>>>(d.echunks, d.ebeg.p, d.aidx.p, d.na_i, d.na, d.C.p, d.CT.p, d.epart.p);
    k_defl_schur<<<1, DT, 0, st>>>(d.nc, d.echunks, d.eext, d.ecell.p, d.epart.p, d.iEjj.p, d.Eje.p, d.Eej.p, d.Ee.p);
    KNP_CUDA(cudaGetLastError());
    d.built_for = p->assembly_id;
}

// The solve is a block's work of 2 us in a kernel of its own of 4. The V-cycle's first kernel does it in
// every block instead where that is less: its grid at most two blocks per SM. The partial sums are few then
// (a chunk per 1,024 nodes and cell: at most 140 with fewer than SOLVE_CELLS cells).
constexpr int SOLVE_ROWS = 152 * 512;

// Most blocks of a gather that runs beside the normalisation: two per SM. With more (some 470 at 75^3) the
// scalars that each of them forms and the second vector that the normalisation then needs cost what the
// launch saves (0.4% of a pass).
constexpr int GATHER_BESIDE = 2 * 152;

bool deflation_gather_beside(const knp_problem* p) { return p->defl->gchunks + p->defl->gext <= GATHER_BESIDE; }

GatherArgs deflation_gather(const knp_problem* p) {
    const Deflation& d = *p->defl;
    GatherArgs a;
    a.nchunks = d.gchunks;
    a.next = d.gext;
    a.cbeg = d.gbeg.p;
    a.cnodes = d.cnodes.p;
    a.N_i = p->N_i;
    a.n = p->n_nodes;
    a.pin = p->pin;
    a.part = d.gpart.p;
    return a;
}

// y = E^{-1} Z^T (s .* v), and what forms s .* v - A Z y and adds Z y. gathered: Z^T (s .* v) is formed
// already; in_vcycle: y may be left to the V-cycle's first kernel
static DeflFuse coarse_solution(knp_problem* p, const double* v, const double* s, bool transpose, const Queue& q,
                                bool gathered, bool in_vcycle) {
    Deflation& d = *p->defl;
    if (!gathered) {
        count_launch();
        launch(k_defl_gather, d.gchunks + d.gext, DT, q, deflation_gather(p), v, s);
    }
    DeflFuse df;
    df.rgrp = d.rgrp.p;
    df.act = d.act.p;
    df.C = transpose ? d.CT.p : d.C.p;
    df.xgrp = d.xgrp.p;
    df.y = d.y.p;
    df.N_i = p->N_i;
    df.pin = p->pin;
    df.ext_group = d.nc;
    df.transpose = transpose;
    df.e.nc = d.nc;
    df.e.nchunks = d.gchunks;
    df.e.next = d.gext;
    df.e.cchunk = d.gcell.p;
    df.e.part = d.gpart.p;
    df.e.iEjj = d.iEjj.p;
    // Z^T A^T Z = E^T: the same Schur complement, E_je and E_ej exchanged
    df.e.Eje = transpose ? d.Eej.p : d.Eje.p;
    df.e.Eej = transpose ? d.Eje.p : d.Eej.p;
    df.e.Ee = d.Ee.p;
    df.solve = in_vcycle && d.nc < SOLVE_CELLS && p->n_nodes <= SOLVE_ROWS;
    if (!df.solve) {
        count_launch();
        launch(k_defl_solve, 1, DT, q, df.e, d.y.p);
    }
    return df;
}

void deflated_vcycle_launch(knp_problem* p, const double* v, const double* s, double* z, bool transpose, double* w,
                            const Queue& q) {
    vcycle_launch(p, v, s, z, coarse_solution(p, v, s, transpose, q, deflation_gather_beside(p), true), w, q);
}

void deflated_precond_apply(knp_problem* p, const double* v, const double* s, double* z, bool transpose,
                            double* w) {
    Deflation& d = *p->defl;
    cudaStream_t st = p->stream;
    const int64_t n = p->n_nodes;
    const bool vcycle = p->amg->inner_cg_max_it == 0;
    const DeflFuse df = coarse_solution(p, v, s, transpose, st, false, vcycle);
    if (vcycle) {
        // one V-cycle: its first kernel forms s .* v - A Z y and its output kernel adds Z y
        vcycle_apply(p, v, s, z, &df, w);
        return;
    }
    if (!d.ones.p) {
        DArray<double> ones;   // kept last, with t there: an allocation may fail
        d.t.alloc(4 * n);
        ones.alloc(4 * n);
        k_fill_ones<<<nbk(4 * n, 256), 256, 0, st>>>(4 * n, ones.p);
        count_launch();
        d.ones = std::move(ones);
    }
    count_launch();
    k_defl_rhs<<<nbk(n, 128), 128, 0, st>>>(n, v, s, df, d.t.p);
    precond_apply(p, d.t.p, d.ones.p, z);
    count_launch();
    k_defl_add<<<nbk(n, 256), 256, 0, st>>>(n, p->N_i, p->pin, d.rgrp.p, d.y.p, d.nc, z);
    KNP_CUDA(cudaGetLastError());
}

}  // namespace knp
