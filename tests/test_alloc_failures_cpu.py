"""A call that runs out of device memory says so, and the call after it finds nothing half built: the
library's own objects linked with a fake CUDA runtime (tests/c/fake_cudart.cpp) whose k-th cudaMalloc fails,
for every k of a call. No GPU."""
import glob
import json
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# One process per scenario. For k = 1, 2, ..., on a problem of its own: the call with its k-th allocation
# failing, the call again, and what that left in use, until no allocation is left to fail.
CHILD = r"""
import ctypes as C, json, sys
from paper_2403_04491_gb300 import knp
lib = knp.load_library(sys.argv[1])
lib.fake_in_use.restype = C.c_size_t
lib.fake_null_launch.restype = C.c_char_p
lib.fake_fail_at.argtypes = [C.c_long]
lib.fake_pending.restype = C.c_long
from synth import make_config
cfg = make_config(1).with_nx(8)

def hierarchy(prob, cg):
    knp._check(lib.fake_identity_hierarchy(prob.handle, cg))

def solve(prob, deflate):
    # zero states and operators: the solver preconditions once (the paper's stopping test) and is done
    prob.assemble_step()
    prob.solve(deflate=deflate, stop_test=knp.KNP_TEST_PAPER)

def coarse_correction():
    def before(prob):
        hierarchy(prob, 1)
        solve(prob, False)
    return before, lambda prob: solve(prob, True), [b"k_defl", b"k_fill_ones", b"k_pcg_init"]

def solver():
    return lambda prob: hierarchy(prob, 1), lambda prob: solve(prob, False), [b"k_pcg"]

def adjoint():
    # the sweep's start, and a look at its (zero) result, whose kernel reads its arrays
    def call(prob):
        prob.adjoint_begin()
        out = (C.c_double * prob.n_dof)()
        p = C.cast(out, C.c_void_p)
        knp._check(lib.knp_adjoint_get(prob.handle, knp.KNP_DEVICE, p, None, None, p))
    return lambda prob: None, call, [b"k_eq42_out"]

def new_hierarchy():
    # in place of one that is there; without a hierarchy a solve is refused
    def after(prob):
        prob.assemble_step()
        try:
            prob.solve()
        except knp.KnpError as e:
            assert e.code == 7, e
        else:
            assert False, "a solve without a hierarchy"
    return lambda prob: hierarchy(prob, 1), lambda prob: hierarchy(prob, 1), [], after

before, call, watch, *after = globals()[sys.argv[2]]()
for w in watch:
    lib.fake_watch(w)
out = []
for k in range(1, 200):
    mesh, prob = knp.problem_from_config(cfg, stream=0)
    before(prob)
    lib.fake_fail_at(k)
    code = 0
    try:
        call(prob)
    except knp.KnpError as e:
        code = e.code
    left = lib.fake_pending()
    lib.fake_fail_at(0)
    if code:
        for f in after:
            f(prob)
    retry = 0
    try:
        call(prob)
    except knp.KnpError as e:
        retry = e.code
    out.append(dict(code=code, retry=retry, null=lib.fake_null_launch().decode(), in_use=lib.fake_in_use()))
    del prob, mesh
    assert lib.fake_in_use() == 0
    if left:
        break
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    from paper_2403_04491_gb300.build import _nvcc, build_library
    objs = glob.glob(os.path.join(os.path.dirname(build_library()), "*.o"))
    if not objs:
        objs = glob.glob(os.path.join(os.path.dirname(build_library(force=True)), "*.o"))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(_nvcc())))), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libknp_fake.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                    "-I", os.path.join(ROOT, "include"), "-I", cuda,
                    os.path.join(ROOT, "tests", "c", "fake_cudart.cpp")] + objs + ["-o", out], check=True)
    return out


def run(fake_library, scenario):
    env = dict(os.environ, PYTHONPATH=ROOT, KNP_NO_GRAPHS="1")
    r = subprocess.run([sys.executable, "-c", CHILD, fake_library, scenario], capture_output=True, text=True, env=env,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])


@pytest.mark.parametrize("scenario", ["coarse_correction", "solver", "adjoint", "new_hierarchy"])
def test_a_failed_allocation_leaves_nothing_half_built(fake_library, scenario):
    runs = run(fake_library, scenario)
    assert len(runs) > 2 and runs[-1]["code"] == 0          # every allocation of the call has failed once
    for k, r in enumerate(runs[:-1], 1):
        assert r["code"] == 3, (k, r)                       # KNP_ERR_OOM
    for k, r in enumerate(runs, 1):
        assert r["retry"] == 0 and r["null"] == "", (k, r)
        assert r["in_use"] == runs[-1]["in_use"], (k, r)
