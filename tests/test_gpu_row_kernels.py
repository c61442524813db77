"""The kernels' choices of lanes, launch and grouping at the sizes where they change.

* operator products with 8, 4 and 1 lanes per row, and with the last block and slice partly empty;
* the V-cycle: symmetric when it smooths equally on both sides;
* time steps from captured graphs against single launches.
"""
import numpy as np
import pytest

from helpers import blockwise_vector_error
from oracle import problem as oproblem, system as osystem
from synth import make_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


# nodes: 284 (8 lanes, a partly empty warp), 4,760 and 4,897 (either side of the 8-lane limit of 4,864),
# 18,768 and 20,448 (either side of the 4-lane limit of 152 * 18 rows per entry of a mean row of 7)
@pytest.mark.parametrize("nx", [15, 67, 68, 135, 141])
def test_operator_products_at_the_lane_limits(nx):
    from paper_2403_04491_gb300 import problem_from_config
    cfg = make_config(1).with_nx(nx)
    pb, s0 = oproblem.from_config(cfg)
    A, _, _ = osystem.assemble(pb, s0)
    _, prob = problem_from_config(cfg)
    prob.assemble_step()
    x = np.random.default_rng(nx).standard_normal(A.shape[0])
    assert blockwise_vector_error(pb, prob.apply_operator(x), A @ x) < 1e-12
    assert blockwise_vector_error(pb, prob.apply_operator_transpose(x), A.T @ x) < 1e-12


# one to four levels. P_0's field blocks are independent, so each is symmetric by itself. The concentrations'
# blocks are mass matrices and some stiffness (condition below 1e3): the dense inverse of the coarsest level is
# symmetric to that times eps, and the rest to some tens of eps. The potentials' are nearly singular (1e9 taken).
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("config,nx", [(1, 20), (1, 32), (1, 97), (4, 256), (2, 11), (2, 29), (2, 48)])
def test_vcycle_is_symmetric(config, nx, precision):
    from paper_2403_04491_gb300 import problem_from_config
    _, prob = problem_from_config(make_config(config).with_nx(nx))
    prob.amg_setup(precision=precision, cheb_degree=2, cheb_degree_pre=2)
    u, v = np.random.default_rng(nx).standard_normal((2, prob.n_dof))
    mu, mv = prob.apply_preconditioner(u), prob.apply_preconditioner(v)
    at = 0
    for n in (prob.N_i, prob.N_e):
        for field in range(4):
            b = slice(at, at + n)
            at += n
            eps = np.finfo(np.float64 if precision == 0 else np.float32).eps
            tol = max(100 * eps, (1e3 if field < 3 else 1e9) * np.finfo(np.float64).eps)
            scale = np.linalg.norm(u[b]) * np.linalg.norm(mv[b]) + np.linalg.norm(v[b]) * np.linalg.norm(mu[b])
            assert np.linalg.norm(mu[b]) > 0
            assert abs(u[b] @ mv[b] - v[b] @ mu[b]) <= tol * scale


# restart 12: several cycles, so that graphs of every basis index are replayed
@pytest.mark.parametrize("config,nx,deflate", [(1, 15, True), (1, 15, False), (2, 13, True), (4, 64, True)])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_graphs_match_single_launches(config, nx, deflate, precision, monkeypatch):
    from paper_2403_04491_gb300 import problem_from_config
    got = {}
    for graphs in (True, False):
        if not graphs:
            monkeypatch.setenv("KNP_NO_GRAPHS", "1")
        _, prob = problem_from_config(make_config(config).with_nx(nx))
        prob.amg_setup(precision=precision)
        prob.step(2, rtol=1e-11, restart=12 if deflate else 30, deflate=deflate)
        s = prob.state_get()
        got[graphs] = [np.concatenate([s["c_i"].ravel(), s["c_e"].ravel()]), np.concatenate([s["phi_i"], s["phi_e"]])]
    # each is within 10 rtol of the solution in the norm of its stopping test (the bar of the parity tests)
    for a, b in zip(got[True], got[False]):
        assert np.linalg.norm(a - b) <= 2 * 10 * 1e-11 * np.linalg.norm(b)
