#pragma once
#include <map>
#include <tuple>
#include <vector>

#include "amg.h"
#include "launch.h"

struct knp_problem;

namespace knp {

constexpr int SOLVE_CELLS = 64;   // the V-cycle's first kernel forms y for fewer cells than this

// Terms of y = E^{-1} g for the arrowhead E of the coarse correction: g = Z^T r as the partial sums part
// (those of cell j at [cchunk[j], cchunk[j + 1]), next of the extracellular space from nchunks on), and
// 1 / E_jj, E_je, E_ej, {E_ee, 1 / Schur complement} (E_je and E_ej exchanged for the transposed operator).
struct CoarseSolve {
    int32_t nc = 0, nchunks = 0, next = 0;
    const int32_t* cchunk = nullptr;
    const double *part = nullptr, *iEjj = nullptr, *Eje = nullptr, *Eej = nullptr, *Ee = nullptr;
};

// The coarse correction's two passes around the V-cycle, done inside it (device pointers and
// scalars; y == nullptr: none). The first kernel of the finest level forms the corrected input
// r - A Z y from r = s .* v (deflate_input.h), and the output kernel adds Z y to the potentials.
struct DeflFuse {
    const int32_t* rgrp = nullptr;   // intracellular node -> its cell group
    const int32_t* act = nullptr;    // node -> active row, -1 where A Z y is zero
    const double* C = nullptr;       // [active rows][8] coefficients of A Z y (or A^T Z y)
    const int32_t* xgrp = nullptr;   // active row -> group on the membrane's other side
    double* y = nullptr;             // [groups + 1] the coarse solution, extracellular group last
    int64_t N_i = 0;
    int32_t pin = -1, ext_group = 0;
    int32_t transpose = 0;           // A^T Z y in place of A Z y
    int32_t solve = 0;               // the first kernel also forms y, from the terms below
    CoarseSolve e;
};

// One captured V-cycle: a CUDA graph instantiated for given arguments (AmgHierarchy::graphs).
struct VcycleGraph {
    cudaGraphExec_t exec = nullptr;
    int launches = 0;
};

struct AmgHierarchy {
    const uint64_t id;   // another for every hierarchy: captured graphs name it, not its address
    int precision = 0;
    int levels = 0;
    std::vector<int64_t> nodes, nnz;
    void* h64 = nullptr;   // AmgDev<double>
    void* h32 = nullptr;   // AmgDev<float>
    // CUDA graphs of single V-cycles, captured on a private stream: per input, scale, output, coarse
    // solution, direction of the coarse correction and the product's w. FGMRES uses them for the first basis
    // vector and, with CG(P_0), for all
    bool use_graphs = true;
    cudaStream_t gstream = nullptr;
    std::map<std::tuple<const double*, const double*, double*, const double*, int, double*>, VcycleGraph> graphs;
    // CG(P_0): P_0^{-1} applied by V-cycle-preconditioned CG per field block (0 = one V-cycle)
    int inner_cg_max_it = 0;
    double inner_cg_rtol = 0.0;
    int64_t inner_its = 0;   // inner CG iterations so far
    // how the hierarchy was built: on the GPU (1) or on the host (0, host_setup), and the rows
    // of P and of the Galerkin products that the GPU setup finished with its long-row kernels
    int setup_on_gpu = 0;
    int64_t long_rows_p = 0, long_rows_rap = 0;
    double setup_ms = 0.0;
    AmgHierarchy();
    ~AmgHierarchy();
};

// degree / pre: Chebyshev steps after / before the coarse-grid correction on every level
void amg_upload(knp_problem* p, const HostHierarchy& H, int precision, int degree, int pre);
struct GpuHierarchy;
// the hierarchy built by amg_build_gpu, taken over on the device (consumes H)
void amg_take_gpu(knp_problem* p, GpuHierarchy& H, int precision, int degree, int pre);
// z = V-cycle(s .* v); with df (y set), z = V-cycle(s .* v - A Z y) + Z y (the coarse correction's
// passes fused into the first and last kernels). With w (allowed if vcycle_forms_w), also the forward
// operator product's w of z.
void vcycle_apply(knp_problem* p, const double* v, const double* s, double* z, const DeflFuse* df = nullptr,
                  double* w = nullptr);
// the same with its kernels launched one by one into q (which may be capturing)
void vcycle_launch(knp_problem* p, const double* v, const double* s, double* z, const DeflFuse& df, double* w,
                   const Queue& q);
// whether z = P_0^{-1} (s .* v) is one V-cycle whose last kernel can form w
bool vcycle_forms_w(const knp_problem* p);
// y = P_0 x with the finest level of the FP64 hierarchy; x, y [n][4] doubles on the device
void p0_apply(knp_problem* p, const double* x, double* y);
// z = P_0^{-1} (s .* v): one V-cycle, or CG(P_0) when the hierarchy was set up for it
void precond_apply(knp_problem* p, const double* v, const double* s, double* z, double* w = nullptr);

}  // namespace knp
