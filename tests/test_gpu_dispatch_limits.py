"""The V-cycle's and the coarse correction's choices of kernel on either side of the sizes where they change.

* the coarse correction against its formula: solved by its own kernel or inside the V-cycle's first one (up to
  63 cells and 77,824 nodes), a cell's sums by a thread or by a warp (more than eight chunks of 1,024 nodes per
  cell), gathers of up to and of more than 304 blocks;
* time and adjoint steps from captured graphs, where the gather runs beside the normalisation (up to 304
  blocks), against single launches, where it never does: the same sums in the same order, so the same bits;
* the V-cycle, symmetric when it smooths equally on both sides, with 8, 4 and 1 lanes per sliced-ELL row, 4 to
  32 lanes per CSR row, 4 to 128 lanes in the restriction and 4 and 1 threads per row of the prolongation.
"""
from dataclasses import replace

import numpy as np
import pytest

from synth import make_config
from synth.mesh import box_cells

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def config(name):
    """(number, intervals per side), or cells of an 8 x 8 array on 100 x 100."""
    if isinstance(name, tuple):
        return make_config(name[0]).with_nx(name[1])
    lo, hi = box_cells(8, 0.08, 0.03, 2)
    return replace(make_config(4), nx=100, cell_lo=lo[:name], cell_hi=hi[:name], _mesh=None)


def coarse_space(mesh, m):
    """Z in the Eq. 4.3 order: a cell's intracellular potentials, and the extracellular ones but the pinned."""
    import scipy.sparse as sp
    nodes_i, nodes_e = mesh.nodes()
    ni, ne = len(nodes_i), len(nodes_e)
    cell = np.zeros(len(m.coords), np.int64)
    for k in range(m.elems.shape[1]):
        cell[m.elems[m.elem_tag > 0, k]] = m.elem_tag[m.elem_tag > 0]
    _, group = np.unique(cell[nodes_i], return_inverse=True)
    nc = group.max() + 1
    ext = np.flatnonzero(nodes_e != mesh.info["pin_vertex"])
    rows = np.concatenate([3 * ni + np.arange(ni), 4 * ni + 3 * ne + ext])
    cols = np.concatenate([group, np.full(len(ext), nc)])
    return sp.csr_matrix((np.ones(len(rows)), (rows, cols)), shape=(4 * (ni + ne), nc + 1))


# The bars are those of the correction's test against the oracle at 16 intervals per side (1e-10, and 1e-8 for
# the exactness on the coarse space), times the intervals over 16: rounding in r - A Z y reaches the coarse
# modes amplified by the ratio of stiffness to membrane capacitance, which grows as 1 / h.
@pytest.mark.parametrize("name", [63, 64, (1, 190), (1, 276), (1, 277), (1, 553), (1, 556), (2, 52), (3, 32)], ids=str)
def test_coarse_correction_is_its_formula(name):
    from paper_2403_04491_gb300 import problem_from_config
    cfg = config(name)
    mesh, prob = problem_from_config(cfg)
    Z = coarse_space(mesh, cfg.mesh)
    prob.amg_setup()
    prob.assemble_step()
    rng = np.random.default_rng(11)
    w, r = rng.standard_normal(Z.shape[1]), rng.standard_normal(prob.n_dof)
    grow = max(1.0, cfg.nx / 16)
    for transpose, A in ((False, prob.apply_operator), (True, prob.apply_operator_transpose)):
        AZ = np.stack([A(np.asarray(Z[:, j].todense()).ravel()) for j in range(Z.shape[1])], axis=1)
        z = prob.apply_deflated_preconditioner(AZ @ w, transpose=transpose)
        assert np.linalg.norm(z - Z @ w) <= 1e-8 * grow * np.linalg.norm(Z @ w)
        y = np.linalg.solve(Z.T @ AZ, Z.T @ r)
        ref = prob.apply_preconditioner(r - AZ @ y) + Z @ y
        z = prob.apply_deflated_preconditioner(r, transpose=transpose)
        assert np.linalg.norm(z - ref) <= 1e-10 * grow * np.linalg.norm(ref)


def both_ways(monkeypatch, cfg, run, **setup):
    """run(problem) with captured graphs and with single launches."""
    from paper_2403_04491_gb300 import problem_from_config
    got = []
    for graphs in (True, False):
        if not graphs:
            monkeypatch.setenv("KNP_NO_GRAPHS", "1")
        _, prob = problem_from_config(cfg)
        prob.amg_setup(**setup)
        got.append(run(prob))
    return got


# restart 12: graphs of every basis index are replayed
@pytest.mark.parametrize("name,restart,setup", [
    ((1, 15), 12, {}), (63, 30, {}), (64, 30, {}), ((1, 190), 30, {}), ((1, 276), 30, {}), ((1, 277), 30, {}),
    ((1, 553), 30, {}), ((1, 556), 30, {}), ((2, 29), 12, {"precision": 1}), ((2, 52), 30, {"precision": 1}),
    ((2, 12), 30, {"inner_cg_max_it": 60, "inner_cg_rtol": 1e-10})], ids=str)
def test_steps_from_graphs_are_those_of_single_launches(monkeypatch, name, restart, setup):
    def run(prob):
        its = [s["iterations"] for s in prob.step(2, rtol=1e-10, restart=restart)]
        return its, prob.state_get()
    (its, a), (its_single, b) = both_ways(monkeypatch, config(name), run, **setup)
    assert its == its_single and min(its) > 1
    for k in ("c_i", "phi_i", "c_e", "phi_e"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("name", [(4, 32), (2, 12), (1, 277)], ids=str)
def test_adjoint_steps_from_graphs_are_those_of_single_launches(monkeypatch, name):
    def run(prob):
        rng = np.random.default_rng(3)
        s = prob.state_get()
        u = np.concatenate([s["c_i"].ravel(), s["phi_i"], s["c_e"].ravel(), s["phi_e"]])
        prob.adjoint_begin()
        its = [prob.adjoint_step(u, rng.standard_normal(prob.n_dof), rtol=1e-10)["iterations"] for _ in range(2)]
        return its, prob.adjoint_get()
    (its, a), (its_single, b) = both_ways(monkeypatch, config(name), run)
    assert its == its_single and min(its) > 1
    for k in a:
        assert np.array_equal(a[k], b[k]), k


# (config, intervals, degree): a single level; sliced-ELL rows by 8, 4 and 1 lanes; the prolongation's two forms on
# either side of 77,824 rows; CSR rows by 16 (4,851 rows of 55 entries, just within the limit), 8, 4 and 32 lanes;
# with P2 elements in 3D also the finest level, whose last step writes the V-cycle's result.
# The concentrations' blocks are mass matrices and some stiffness (condition below 1e3): the dense inverse of the
# coarsest level is symmetric to that times eps, the rest to some tens of eps. The potentials are probed
# orthogonally to their nearly constant modes, where the blocks' condition is at most of the order of the number of
# nodes (in FP32, whose rounding that would drown, only the concentrations are).
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("number,nx,degree", [(1, 15, 1), (1, 67, 1), (1, 68, 1), (1, 276, 1), (1, 277, 1),
                                               (2, 16, 1), (2, 36, 1), (2, 40, 1), (2, 48, 1), (2, 10, 2), (2, 16, 2)])
def test_vcycle_is_symmetric_beside_its_constants(number, nx, degree, precision):
    from paper_2403_04491_gb300 import problem_from_config
    mesh, prob = problem_from_config(make_config(number).with_nx(nx), degree=degree)
    prob.amg_setup(precision=precision, cheb_degree=2, cheb_degree_pre=2)
    nodes_e = mesh.p2()["nodes_e"] if degree == 2 else mesh.nodes()[1]
    free = [np.ones(prob.N_i, bool), nodes_e != mesh.info["pin_vertex"]]     # P2 nodes: the vertices come first
    u, v = np.random.default_rng(nx).standard_normal((2, prob.n_dof))
    at = 0
    blocks = []
    for region, n in enumerate((prob.N_i, prob.N_e)):
        for field in range(4):
            b = slice(at, at + n)
            at += n
            if field == 3:
                for x in (u, v):
                    x[b] = np.where(free[region], x[b] - x[b][free[region]].mean(), 0.0)
            blocks.append((b, field))
    mu, mv = prob.apply_preconditioner(u), prob.apply_preconditioner(v)
    for b, field in blocks:
        if field == 3 and precision == 1:
            continue
        eps = np.finfo(np.float64 if precision == 0 else np.float32).eps
        tol = 100 * eps * (prob.N_i + prob.N_e) if field == 3 else max(100 * eps, 1e3 * np.finfo(np.float64).eps)
        scale = np.linalg.norm(u[b]) * np.linalg.norm(mv[b]) + np.linalg.norm(v[b]) * np.linalg.norm(mu[b])
        assert np.linalg.norm(mu[b]) > 0
        assert abs(u[b] @ mv[b] - v[b] @ mu[b]) <= tol * scale, (b, field)
