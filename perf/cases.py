"""Timed cases of the KNP-EMI step library: what a program that uses it calls, and on what.

One pass of a case starts from a state on the device and goes through the public entry points:

* ``step``     knp_state_set, knp_step over a few time steps (membrane update, assembly, FGMRES with
               the AMG V-cycle), knp_state_get: a simulation's time loop between two looks at its state;
* ``adjoint``  knp_adjoint_begin, then for each reverse step knp_state_set and knp_adjoint_step,
               then knp_adjoint_get: the reverse sweep of a checkpointed segment;
* ``rebuild``  knp_state_set, knp_assemble_step, knp_amg_setup on the assembled operator, knp_solve: the
               time-dependent preconditioner P_n (Eq. 4.4), a hierarchy set up for one step.

The mesh, the problem and the P_0 hierarchy (built from the problem's own uniform initial state) are what
a program lays out once and keeps, so all states of one case share them; a state holds its own fields.
States are smooth perturbations of the physiological rest values, electroneutral (Cl = Na + K).

``exact`` restates the step and its adjoint in dense 64-bit torch (P1 elements, up to 12,000 unknowns).
"""
import ctypes
import itertools
import math

import numpy as np
import torch

import paper_2403_04491_gb300 as knp
from paper_2403_04491_gb300.knp import KNP_DEVICE, load_library

# Table 2 of the paper (SI units)
R, T, F, CM = 8.314, 300.0, 9.648e4, 0.02
Z = (1.0, 1.0, -1.0)
D = (1.33e-9, 1.96e-9, 2.03e-9)
C_I0, C_E0 = (12.0, 125.0, 137.0), (100.0, 4.0, 104.0)
PHI_M0, PHI_REST = -67.74e-3, -65e-3
GBAR_NA, GBAR_K = 1200.0, 360.0
W0 = (0.276, 0.0379, 0.688)
PUMP, P_NA, P_K = 1.115e-6, 10.0, 1.5
N_ODE = 25
LENGTH = 100e-6
LEAK, HH, KIR = 0, 1, 2
MODELS = {"leak": LEAK, "hh": HH, "kir": KIR}
G_LEAK = {"leak": (0.2, 0.8, 0.0), "hh": (0.2, 0.8, 0.0), "kir": (1.0, 4.0, 0.0)}
DT = {"leak": 1e-4, "hh": 5e-5, "kir": 1e-4}
STIM_G, STIM_T1, STIM_X = 40.0, 1e-3, 0.4 * LENGTH      # membrane stimulus of the HH workloads
SOURCE, SOURCE_T1, SOURCE_X = (-1.0, 1.0, 0.0), 2.05e-3, 0.5 * LENGTH   # bulk source of the Kir workloads
EXACT_DOF = 12000
# Relative tolerance of every solve. At looser ones, whether the stopping test passes one iteration
# earlier or later can hang on the last bits of a sum, and the states of two equally good builds then
# differ by the tolerance itself.
RTOL = 1e-11


def _case(name, kind, nx, ny, nz, cells, model, fp32, steps, degree=1, refine=False):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, cells=cells, model=model, fp32=fp32, steps=steps, degree=degree,
             refine=refine)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest workload: one cell in 2D, 4,612 unknowns; launches and latency
        _case("step-2d-32", "step", 32, 32, 0, 1, "leak", False, 3),
        # 2D Kir-Na/K membrane with a bulk source on an odd, non-square grid
        _case("step-2d-kir-97x75", "step", 97, 75, 0, 1, "kir", False, 3),
        # the 16-cell 2D workload at full size (its forward run), 274,052 unknowns
        _case("step-2d-256-16cells", "step", 256, 256, 0, 4, "leak", False, 2),
        # a small ragged 3D grid with HH channels, FP64 hierarchy
        _case("step-3d-33x29x27", "step", 33, 29, 27, 1, "hh", False, 3),
        # interface-refined tensor grid (32^3 -> 44^3), anisotropic elements, 372,284 unknowns
        _case("step-3d-refined-32", "step", 32, 32, 32, 1, "hh", False, 2, refine=True),
        # the plain FP64 3D workload, 1,114,732 unknowns
        _case("step-3d-64", "step", 64, 64, 64, 1, "hh", False, 2),
        # mixed precision (FP32 hierarchy under FP64 FGMRES), 27 cells on an odd grid, 1.9M unknowns
        _case("step-3d-75-27cells-fp32", "step", 75, 75, 75, 3, "hh", True, 2),
        # the 125-cell mixed-precision workload, 9,317,836 unknowns: the largest
        _case("step-3d-128-125cells-fp32", "step", 128, 128, 128, 5, "hh", True, 2),
        # P2 elements in 3D: longer rows of uneven length
        _case("step-3d-p2-20", "step", 20, 20, 20, 1, "hh", False, 2, degree=2),
        # reverse sweep of the 2D differentiation workload
        _case("adjoint-2d-256-16cells", "adjoint", 256, 256, 0, 4, "leak", False, 2),
        # reverse sweep in 3D with HH gates
        _case("adjoint-3d-40", "adjoint", 40, 40, 40, 1, "hh", False, 2),
        # preconditioner rebuilt for the step (P_n), mixed precision
        _case("rebuild-3d-48-fp32", "rebuild", 48, 48, 48, 1, "hh", True, 1),
    ]


def draw(rng):
    """Dimension, direction, membrane, precision, degree and sizes (over their logarithm, odd and
    unequal ones included) of the listed range."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("step", "step", "step", "step", "adjoint", "rebuild"))
        model = rng.choice(("leak", "hh", "hh") if kind == "adjoint" else ("leak", "hh", "hh", "kir"))
        dim = rng.choice((2, 3, 3))
        degree = 2 if kind == "step" and rng.random() < 0.15 else 1
        fp32 = kind != "adjoint" and rng.random() < 0.4
        top = {(2, 1): 320, (2, 2): 128, (3, 1): 120, (3, 2): 24}[dim, degree]
        if kind != "step":
            top = min(top, 256 if dim == 2 else 56)
        low = 20 if dim == 2 else 12
        n = [int(round(math.exp(rng.uniform(math.log(low), math.log(top)))))] * dim
        if rng.random() < 0.5:
            n = [min(top, max(low, int(round(v * rng.uniform(0.8, 1.2))))) for v in n]
        cells = rng.choice([c for c in (1, 1, 2, 3, 4, 5) if c == 1 or min(n) >= 10 * c])
        refine = dim == 3 and degree == 1 and cells == 1 and max(n) <= 32 and rng.random() < 0.25
        case = _case(None, kind, n[0], n[1], n[2] if dim == 3 else 0, cells, model, fp32, rng.choice((1, 2, 3)),
                     degree, refine)
        if _cost(case) <= 0.7 * most:
            return case


def _cost(case):
    """Time of a pass up to a factor: bytes and FP64 operations at the card's rates."""
    w = work(case)
    return max(w["bytes"] / 6.8e12, w["flops"] / 1.1e12)


# ---------------------------------------------------------------- mesh (structured, Model-A shaped)

def _cell_faces(n, cells, dim):
    """Lower and upper grid plane of each cell along one axis of n intervals."""
    if cells == 1:
        lo, hi = ((0.25,), (0.75,)) if dim == 2 else ((0.3,), (0.7,))
    else:
        side, gap = 0.6 / cells, 0.2 / cells
        start = 0.5 - 0.5 * (cells * side + (cells - 1) * gap)
        lo = [start + i * (side + gap) for i in range(cells)]
        hi = [v + side for v in lo]
    snap = lambda v: np.floor(np.asarray(v) * n + 0.5).astype(np.int64)
    return snap(lo), snap(hi)


def _mesh(case):
    """Vertices, simplices (2 triangles or 6 Kuhn tetrahedra per grid box) and cell tags."""
    n = [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])
    dim = len(n)
    axes, faces = [], []
    for m in n:
        lo, hi = _cell_faces(m, case["cells"], dim)
        plane, at = [0.0], [0]
        for i in range(m):
            near = case["refine"] and np.any(np.abs(i + 0.5 - np.concatenate([lo, hi])) <= 1)
            k = 4 if near else 1
            plane += [(i + j / k) / m * LENGTH for j in range(1, k + 1)]
            at.append(len(plane) - 1)
        axes.append(np.array(plane))
        faces.append((np.array(at)[lo], np.array(at)[hi]))
    n1 = [len(a) for a in axes]
    coords = np.stack([g.reshape(-1) for g in np.meshgrid(*axes[::-1], indexing="ij")][::-1], axis=1)
    stride = np.cumprod([1] + n1[:-1])
    base = sum(g.reshape(-1) for g in
               np.meshgrid(*[np.arange(m - 1, dtype=np.int32) * s for m, s in zip(n1, stride)][::-1], indexing="ij"))
    paths = [np.cumsum([0] + [stride[a] for a in perm]) for perm in itertools.permutations(range(dim))]
    elems = (base[:, None, None] + np.array(paths, dtype=np.int32)[None]).reshape(-1, dim + 1).astype(np.int32)
    tag = np.zeros([m - 1 for m in n1[::-1]], np.int32)
    for j, box in enumerate(itertools.product(range(case["cells"]), repeat=dim)):
        tag[tuple(slice(int(faces[a][0][box[a]]), int(faces[a][1][box[a]])) for a in range(dim))[::-1]] = j + 1
    return coords, elems, np.repeat(tag.reshape(-1), len(paths))


def _facet_leak(case, n_facets):
    """Per-facet leak conductances; the leak workloads vary g_K per facet (log-normal, sigma 0.2)."""
    g = np.tile(np.array(G_LEAK[case["model"]]), (n_facets, 1))
    if case["model"] == "leak":
        g[:, 1] *= np.exp(0.2 * np.random.default_rng(1).standard_normal(n_facets))
    return g


# ---------------------------------------------------------------- what a program keeps

class Kept:
    """Mesh, problem and P_0 hierarchy of a case, and where its nodes are."""

    def __init__(self, case):
        coords, elems, tag = _mesh(case)
        self.mesh = knp.Mesh(coords, elems, tag)
        verts = self.mesh.facets()[0]
        n_facets = len(verts)
        if case["degree"] == 2:
            p2 = self.mesh.p2()
            points = np.vstack([coords, 0.5 * (coords[p2["edges"][:, 0]] + coords[p2["edges"][:, 1]])])
            nodes_i, nodes_e, nodes_m = p2["nodes_i"], p2["nodes_e"], p2["membrane_nodes"]
        else:
            points = coords
            nodes_i, nodes_e = self.mesh.nodes()
            nodes_m = np.unique(verts)
        kir, hh = case["model"] == "kir", case["model"] == "hh"
        source = (points[:, 0] < SOURCE_X)[:, None] * np.array(SOURCE)[None] if kir else None
        self.problem = knp.Problem(self.mesh, dict(
            n_ions=3, z=Z, D_i=D, D_e=D, R=R, T=T, F=F, Cm=CM, dt=DT[case["model"]], c_i0=C_I0, c_e0=C_E0,
            phi_M0=PHI_M0, facet_model=np.full(n_facets, MODELS[case["model"]]),
            facet_gleak=_facet_leak(case, n_facets), gbar_na=GBAR_NA, gbar_k=GBAR_K, phi_rest=PHI_REST, w0=W0,
            n_ode=N_ODE, stim_kind=int(hh), stim_gbar=STIM_G, stim_t0=0.0, stim_t1=STIM_T1,
            stim_mask=(coords[verts][:, :, 0].mean(axis=1) < STIM_X), rho_pump=PUMP, P_na=P_NA, P_k=P_K,
            source_e=source, source_t0=0.0, source_t1=SOURCE_T1, degree=case["degree"]))
        self.problem.amg_setup(precision=int(case["fp32"]))
        at = lambda v: torch.as_tensor(points[v] / LENGTH, device="cuda")
        self.at_i, self.at_e, self.at_m, self.n_facets = at(nodes_i), at(nodes_e), at(nodes_m), n_facets


_kept = {}


def _keep(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _kept:
        _kept.clear()
        _kept[key] = Kept(case)
    return _kept[key]


def _wave(rng, at):
    """A smooth field of values in [-1, 1]: three plane waves of random direction and phase."""
    f = torch.zeros(len(at), dtype=torch.float64, device=at.device)
    for _ in range(3):
        k = torch.as_tensor(rng.uniform(-6.0, 6.0, at.shape[1]), device=at.device)
        f += torch.cos(at @ k + rng.uniform(0.0, 2.0 * math.pi)) / 3.0
    return f


def _fields(rng, at_i, at_e, at_m):
    """One state: c [c_i (3 N_i), c_e (3 N_e)], phi [phi_i, phi_e], gates w [3, n_m]."""
    c = []
    for at, c0 in ((at_i, C_I0), (at_e, C_E0)):
        na, k = (c0[q] * (1.0 + 0.02 * _wave(rng, at)) for q in (0, 1))
        c += [na, k, na + k]
    phi = torch.cat([PHI_M0 + 2e-3 * _wave(rng, at_i), 1e-4 * _wave(rng, at_e)])
    w = torch.stack([g * (1.0 + 0.05 * _wave(rng, at_m)) for g in W0])
    return dict(c=torch.cat(c), phi=phi, w=w)


def _inputs(case, seed, at_i, at_e, at_m):
    """States u_0 .. u_steps of a segment (the first one alone for a forward pass) and, for the
    adjoint, the loss derivative of each later state: probes of every field, as a data fit has."""
    rng = np.random.default_rng(seed)
    states = [_fields(rng, at_i, at_e, at_m)]
    loss = []
    if case["kind"] == "adjoint":
        other = _fields(rng, at_i, at_e, at_m)
        n_i, n = len(at_i), len(at_i) + len(at_e)
        for s in range(1, case["steps"] + 1):
            states.append({k: (1.0 - 0.02 * s) * v + 0.02 * s * other[k] for k, v in states[0].items()})
            g = torch.zeros(4 * n, dtype=torch.float64, device=at_i.device)
            probe = torch.as_tensor(rng.choice(4 * n, 64 + n // 64, replace=False), device=at_i.device)
            scale = torch.ones_like(g)
            scale[3 * n_i:4 * n_i] = scale[4 * n_i + 3 * (n - n_i):] = 1e3      # volts against mol/m^3
            g[probe] = torch.as_tensor(rng.standard_normal(len(probe)), device=at_i.device) * scale[probe]
            loss.append(g)
    return states, loss


def _eq43(s, n_i, n_e):
    """A state as one vector in the Eq. 4.3 order [c_i, phi_i, c_e, phi_e]."""
    return torch.cat([s["c"][:3 * n_i], s["phi"][:n_i], s["c"][3 * n_i:], s["phi"][n_i:]])


# ---------------------------------------------------------------- one pass

def prepare(case, seed):
    kept = _keep(case)
    states, loss = _inputs(case, seed, kept.at_i, kept.at_e, kept.at_m)
    p = kept.problem
    out = {k: torch.empty_like(v) for k, v in states[0].items()}
    if case["kind"] == "adjoint":
        out = dict(dLdu0=torch.empty(p.n_dof, dtype=torch.float64, device="cuda"),
                   dLdw0=torch.empty(3, p.n_mv, dtype=torch.float64, device="cuda"),
                   grad_gleak=torch.empty(kept.n_facets, 3, dtype=torch.float64, device="cuda"),
                   lam=torch.empty(p.n_dof, dtype=torch.float64, device="cuda"))
    return dict(case=case, kept=kept, states=states, u=[_eq43(s, p.N_i, p.N_e) for s in states], loss=loss, out=out)


def _ptr(t, offset=0):
    return ctypes.cast(ctypes.c_void_p(t.data_ptr() + 8 * offset), ctypes.POINTER(ctypes.c_double))


def _parts(p, s):
    return (_ptr(s["c"]), _ptr(s["phi"]), _ptr(s["c"], 3 * p.N_i), _ptr(s["phi"], p.N_i), _ptr(s["w"]))


def _check(code):
    if code:
        raise RuntimeError(load_library().knp_last_error().decode())


def run(state):
    lib, case, p, out = load_library(), state["case"], state["kept"].problem, state["out"]
    set_state = lambda s, t: _check(lib.knp_state_set(p.handle, KNP_DEVICE, *_parts(p, s), t))
    dt = DT[case["model"]]
    if case["kind"] == "adjoint":
        p.adjoint_begin()
        for n in range(case["steps"], 0, -1):
            set_state(state["states"][n - 1], (n - 1) * dt)
            p.adjoint_step(state["u"][n], state["loss"][n - 1], rtol=RTOL)
        at = lambda k: ctypes.c_void_p(out[k].data_ptr())
        _check(lib.knp_adjoint_get(p.handle, KNP_DEVICE, at("dLdu0"), at("dLdw0"), at("grad_gleak"), at("lam")))
        return out
    set_state(state["states"][0], 0.0)
    if case["kind"] == "rebuild":
        for _ in range(case["steps"]):
            p.assemble_step()
            p.amg_setup(precision=int(case["fp32"]))
            p.solve(rtol=RTOL)
    else:
        p.step(case["steps"], rtol=RTOL)
    _check(lib.knp_state_get(p.handle, KNP_DEVICE, *_parts(p, out), None))
    return out


def work(case):
    """Bytes and FP64 operations that the method needs per pass, from the grid's counts: per FGMRES
    iteration the operator and the smoother's three passes over the finest level once each, the Krylov
    vectors twice, with the about 24 iterations that this tolerance takes."""
    dim = 3 if case["nz"] else 2
    n = float(np.prod([v + 1 for v in (case["nx"], case["ny"], case["nz"] or 0)]))
    row = {(2, 1): 7.0, (3, 1): 14.5, (2, 2): 11.5, (3, 2): 27.0}[dim, case["degree"]]
    n *= 1.05 * (1.0 if case["degree"] == 1 else 2.0 ** dim) * (2.5 if case["refine"] else 1.0)
    its, word = 24.0, 4.0 if case["fp32"] else 8.0
    operator = n * (row * 60.0 + 144.0)
    smoother = 3.0 * n * (row * (4.0 + 4.0 * word) + 24.0 * word)
    krylov = 2.0 * (0.5 * its + 2.0) * n * 32.0
    flops = n * (14.0 * row + 26.0 + 4.0 * 4.0 * (0.5 * its + 1.0) + (0.0 if case["fp32"] else 24.0 * row))
    return dict(bytes=case["steps"] * (its * (operator + smoother + krylov) + 3.0 * operator),
                flops=case["steps"] * its * flops)


# ---------------------------------------------------------------- the same in dense 64-bit torch

class Dense:
    """The P1 discretisation of a case (Sections 3.2, 3.3, 4.1) and its linearised step as dense
    matrices. Unknowns in the Eq. 4.3 order; the phi_e of the node nearest to the origin is pinned."""

    def __init__(self, case):
        self.case, self.dt = case, DT[case["model"]]
        coords, elems, tag = _mesh(case)
        dim = self.dim = coords.shape[1]
        inside = tag > 0
        on = [np.unique(elems[m]) for m in (inside, ~inside)]
        loc = [np.full(len(coords), -1, np.int64) for _ in on]
        for l, v in zip(loc, on):
            l[v] = np.arange(len(v))
        self.n = [len(v) for v in on]
        # membrane facets: shared by an inside and an outside element, sorted
        local = [[c for c in range(dim + 1) if c != s] for s in range(dim + 1)]
        fac = np.sort(elems[:, local], axis=2)
        both = [np.unique(fac[m].reshape(-1, dim), axis=0) for m in (inside, ~inside)]
        allf = np.concatenate(both)
        facets, count = np.unique(allf, axis=0, return_counts=True)
        facets = facets[count == 2]
        mv = np.unique(facets)
        t = lambda a: torch.as_tensor(a, device="cuda")
        self.at = [t(coords[v] / LENGTH) for v in on + [mv]]
        self.mv = [t(l[mv]) for l in loc]
        self.fm = t(np.searchsorted(mv, facets))
        self.stim = t((coords[facets][:, :, 0].mean(axis=1) < STIM_X).astype(float))
        self.gleak = t(_facet_leak(case, len(facets)))
        e = coords[facets][:, 1:] - coords[facets][:, :1]
        gram = np.einsum("fix,fjx->fij", e, e)
        self.area = t(np.sqrt(np.linalg.det(gram)) / math.factorial(dim - 1))
        self.pin = int(np.argmin((coords[on[1]] ** 2).sum(axis=1)))
        # element mass and stiffness per region
        self.region = []
        for m, l in zip((inside, ~inside), loc):
            x = coords[elems[m]]
            J = x[:, 1:] - x[:, :1]
            G = np.linalg.inv(J).transpose(0, 2, 1)
            G = np.concatenate([-G.sum(axis=1, keepdims=True), G], axis=1)
            vol = np.abs(np.linalg.det(J)) / math.factorial(dim)
            mass = vol[:, None, None] * (np.ones((dim + 1, dim + 1)) + np.eye(dim + 1)) / ((dim + 1) * (dim + 2))
            self.region.append((t(l[elems[m]]), t(mass), t(vol[:, None, None] * np.einsum("njx,nlx->njl", G, G))))
        self.source = t((coords[on[1]][:, 0] < SOURCE_X).astype(float))
        # moments of lambda_a lambda_b (lambda_c) over a unit facet
        mom = lambda *ids: math.factorial(dim - 1) / math.factorial(dim - 1 + len(ids)) * math.prod(
            math.factorial(ids.count(a)) for a in range(dim))
        r = range(dim)
        self.m2 = t(np.array([[mom(a, b) for b in r] for a in r]))
        self.m3 = t(np.array([[[mom(a, b, c) for c in r] for b in r] for a in r]))

    def membrane(self, c, phi, w):
        """C_r^k, phi_M, the new gates and the channel currents' nodal factors at the membrane nodes."""
        z, d = (torch.tensor(v, dtype=torch.float64, device="cuda")[:, None] for v in (Z, D))
        cm = [c[r][:, self.mv[r]] for r in (0, 1)]
        phi_m = phi[0][self.mv[0]] - phi[1][self.mv[1]]
        coef = [(d * z * z * v) / (d * z * z * v).sum(0) * CM / (F * z) for v in cm]
        drive = phi_m - R * T / (F * z) * torch.log(cm[1] / cm[0])
        v = 1e3 * (phi_m - PHI_REST)
        trap = lambda x: torch.where(x.abs() < 1e-6, 1.0 - x / 2.0 + x * x / 12.0,
                                     torch.where(x.abs() < 1e-6, torch.ones_like(x), x)
                                     / torch.expm1(torch.where(x.abs() < 1e-6, torch.ones_like(x), x)))
        a = torch.stack([0.1 * trap((10.0 - v) / 10.0), trap((25.0 - v) / 10.0), 0.07 * torch.exp(-v / 20.0)])
        b = torch.stack([0.125 * torch.exp(-v / 80.0), 4.0 * torch.exp(-v / 18.0),
                         1.0 / (torch.exp((30.0 - v) / 10.0) + 1.0)])
        end = a / (a + b)
        w = end + (w - end) * torch.exp(-(a + b) * 1e3 * self.dt)
        return cm, coef, phi_m, drive, w

    def system(self, c, phi, w, gleak, time):
        """Entries (row, column, value) of A_{n-1}, f_n and w_n from the state (c, phi per region, w)."""
        model, dt, psi = self.case["model"], self.dt, R * T / F
        cm, coef, phi_m, drive, w = self.membrane(c, phi, w)
        nodal = [gleak[:, k, None] * drive[k][self.fm] for k in range(3)]
        if model == "hh":
            stim = STIM_G if time < STIM_T1 else 0.0
            nodal[0] = nodal[0] + (stim * self.stim)[:, None] * drive[0][self.fm]
            nodal[0] = nodal[0] + GBAR_NA * (w[1] ** 3 * w[2] * drive[0])[self.fm]
            nodal[1] = nodal[1] + GBAR_K * (w[0] ** 4 * drive[1])[self.fm]
        if model == "kir":
            ek0 = psi * math.log(C_E0[1] / C_I0[1])
            fk = ((1.0 + math.exp(0.433)) * (1.0 + math.exp(-(0.1186 + ek0) / 0.0441))
                  / (1.0 + torch.exp((drive[1] + 0.0185) / 0.0425)) / (1.0 + torch.exp(-(0.1186 + phi_m) / 0.0441))
                  * torch.sqrt(cm[1][1] / C_E0[1]))
            na = cm[0][0] ** 1.5
            j = (PUMP * na / (na + P_NA ** 1.5) * cm[1][1] / (cm[1][1] + P_K))[self.fm]
            nodal[0] = nodal[0] + 3.0 * F * j
            nodal[1] = gleak[:, 1, None] * (drive[1] * fk)[self.fm] - 2.0 * F * j
        n, first = self.n, (0, 4 * self.n[0])
        rows, cols, vals = [], [], []
        f = torch.zeros(4 * sum(n), dtype=torch.float64, device="cuda")

        def put(r0, rn, c0, cn, v):
            shape = v.shape
            rows.append((r0 + rn)[:, :, None].expand(shape).reshape(-1))
            cols.append((c0 + cn)[:, None, :].expand(shape).reshape(-1))
            vals.append(v.reshape(-1))

        for r in (0, 1):
            q, sign, o, oq = 1 - r, (1.0, -1.0)[r], first[r], first[1 - r]
            el, mass, stiff = self.region[r]
            mine, other = self.mv[r][self.fm], self.mv[q][self.fm]
            for k in range(3):
                tau = dt * D[k]
                put(o + k * n[r], el, o + k * n[r], el, mass + tau * stiff)
                put(o + 3 * n[r], el, o + k * n[r], el, Z[k] * tau * stiff)
                drift = tau * Z[k] / psi * c[r][k][el].mean(dim=1)[:, None, None] * stiff
                cmass = self.area[:, None, None] * torch.einsum("fa,ajl->fjl", coef[r][k][self.fm], self.m3)
                for row, s in ((o + k * n[r], 1.0), (o + 3 * n[r], Z[k])):
                    put(row, el, o + 3 * n[r], el, s * drift)
                    put(row, mine, o + 3 * n[r], mine, s * cmass)
                    put(row, mine, oq + 3 * n[q], other, -s * cmass)
                load = self.area[:, None] * (nodal[k] @ self.m2)
                cap = self.area[:, None] * torch.einsum("fa,fb,abj->fj", coef[r][k][self.fm], phi_m[self.fm], self.m3)
                old = c[r][k]
                if model == "kir" and r == 1 and 0.0 < time + dt <= SOURCE_T1:
                    old = old + dt * SOURCE[k] * self.source
                f = f.index_add(0, (o + k * n[r] + el).reshape(-1), torch.einsum("tjl,tl->tj", mass, old[el]).reshape(-1))
                f = f.index_add(0, (o + k * n[r] + mine).reshape(-1),
                                (-sign * (dt * load / (F * Z[k]) - cap)).reshape(-1))
                f = f.index_add(0, (o + 3 * n[r] + mine).reshape(-1), (-sign * dt * load / F).reshape(-1))
            cap = self.area[:, None] * (phi_m[self.fm] @ self.m2) * CM / F
            f = f.index_add(0, (o + 3 * n[r] + mine).reshape(-1), (sign * cap).reshape(-1))
        rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        pin = first[1] + 3 * n[1] + self.pin
        free = ((rows != pin) & (cols != pin)).double()
        keep = torch.ones_like(f)
        keep[pin] = 0.0
        return rows, cols, vals * free, f * keep, w, pin

    def solve(self, rows, cols, vals, f, pin, transpose=False):
        """Dense LU with symmetric diagonal scaling and two steps of refinement."""
        N = len(f)
        A = torch.zeros(N * N, dtype=torch.float64, device="cuda")
        A.index_add_(0, (cols * N + rows) if transpose else (rows * N + cols), vals.detach())
        A = A.view(N, N)
        A[pin, pin] = 1.0
        s = A.diagonal().abs().rsqrt()
        A *= s[:, None]
        A *= s[None, :]
        lu, piv = torch.linalg.lu_factor(A)
        b = f.detach() * s
        x = torch.linalg.lu_solve(lu, piv, b[:, None])
        for _ in range(2):
            x = x + torch.linalg.lu_solve(lu, piv, b[:, None] - A @ x)
        return x[:, 0] * s

    def split(self, u):
        n, m = self.n, 4 * self.n[0]
        return ([u[:3 * n[0]].view(3, -1), u[m:m + 3 * n[1]].view(3, -1)], [u[3 * n[0]:m], u[m + 3 * n[1]:]])


def exact(case, seed):
    # at most this many unknowns: the count for a cell of the domain's full width (an upper bound)
    bound = 4 * np.prod([v + 1 for v in (case["nx"], case["ny"], case["nz"] or 0)]) * 1.3
    if case["degree"] != 1 or case["refine"] or bound > EXACT_DOF:
        return None
    d = Dense(case)
    states, loss = _inputs(case, seed, *d.at)
    if case["kind"] != "adjoint":
        u, w, time = _eq43(states[0], *d.n), states[0]["w"], 0.0
        for _ in range(case["steps"]):
            c, phi = d.split(u)
            rows, cols, vals, f, w, pin = d.system(c, phi, w, d.gleak, time)
            u = d.solve(rows, cols, vals, f, pin)
            time += d.dt
        c, phi = d.split(u)
        return dict(c=torch.cat([v.reshape(-1) for v in c]), phi=torch.cat(phi), w=w)
    rho = torch.zeros_like(loss[0])
    gam = torch.zeros_like(states[0]["w"])
    grad = torch.zeros_like(d.gleak)
    for n in range(case["steps"], 0, -1):
        u = _eq43(states[n - 1], *d.n).requires_grad_()
        w, g = states[n - 1]["w"].clone().requires_grad_(), d.gleak.clone().requires_grad_()
        rows, cols, vals, f, w_new, pin = d.system(*d.split(u), w, g, (n - 1) * d.dt)
        rhs = loss[n - 1] + rho
        lam = d.solve(rows, cols, vals, rhs, pin, transpose=True)
        u_n = _eq43(states[n], *d.n)
        form = (lam * f).sum() - (lam[rows] * vals * u_n[cols]).sum() + (gam * w_new).sum()
        rho, gam, more = torch.autograd.grad(form, (u, w, g), allow_unused=True)
        gam = torch.zeros_like(w) if gam is None else gam
        grad = grad + more
    return dict(dLdu0=rho, dLdw0=gam, grad_gleak=grad, lam=lam)
