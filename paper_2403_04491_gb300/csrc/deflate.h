// Coarse correction of the potentials' near-null modes around P_0^{-1} (deflate.cu).
#pragma once
#include "deflate_input.h"
#include "problem.h"

namespace knp {
// Forms the per-step data of the correction (row sums of the membrane terms, the arrowhead
// E = Z^T A Z) from the current assembly; does nothing if it is already current.
void deflation_prepare(knp_problem* p);
// z = P_0^{-1} (r - A Z y) + Z y with r = s .* v, y = E^{-1} Z^T r (after deflation_prepare); with
// transpose, A^T and E^T in their places (P_0 is symmetric)
void deflated_precond_apply(knp_problem* p, const double* v, const double* s, double* z, bool transpose = false,
                            double* w = nullptr);
// what forms Z^T r's partial sums (after deflation_prepare), and whether the kernel that normalises r does
GatherArgs deflation_gather(const knp_problem* p);
bool deflation_gather_beside(const knp_problem* p);
// the same with one V-cycle as P_0^{-1}, its kernels launched one by one into q (which may be capturing);
// with deflation_gather_beside the partial sums of Z^T r are there already
void deflated_vcycle_launch(knp_problem* p, const double* v, const double* s, double* z, bool transpose, double* w,
                            const Queue& q);
void deflation_free(Deflation* d);
}  // namespace knp
