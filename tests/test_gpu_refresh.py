"""Numeric-only refreshes of the hierarchies: the Galerkin values at the state of
the refresh, from that state's own matrix, bit for bit."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import amg as oamg
from synthetic import make_problem

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def levels(s, w):
    return [s.export_level(w, l) for l in range(s.hierarchy_info(w)[0].size)]


@pytest.mark.parametrize("opts", [{}, dict(schur=2), dict(schur=3), dict(precision=1, interp_S=1)])
def test_second_newton_iteration_refreshes_from_its_own_matrix(opts):
    """Two Newton iterations with structure reuse refresh once, at the state after
    the first. A context that assembles and builds there has that state's level-0
    values; every refreshed Galerkin operator is the product of the factors of the
    first build with them, and differs from the first build's."""
    prob = make_problem("tiny", shape=(20, 18, 10), seed=11, dt_days=0.5)
    args = (prob["p_n"], prob["T_n"], prob["dt"])
    newton = dict(tol_f=0.0, tol_dx=0.0, rtol=1e-12, reuse=True, coarse_size=40, **opts)
    new = lambda: thermo.Solver.from_problem(prob)
    first, second, fresh, start = new(), new(), new(), new()
    p, T, _ = first.newton_step(*args, max_newton=1, **newton)
    second.newton_step(*args, max_newton=2, **newton)
    for s, state in ((fresh, (p, T)), (start, args[:2])):
        s.assemble(*state, prob["p_n"], prob["T_n"], prob["dt"])
        s.build(coarse_size=40, **opts)
    for w in (0, 1):
        old, got, A0 = levels(start, w), levels(second, w), levels(fresh, w)[0]["A"]
        assert len(got) == len(old) > 2
        A = A0
        for l, (a, b) in enumerate(zip(old, got)):
            if l > 0:
                assert all(np.array_equal(x, y) for x, y in zip(b["A"], A)), (w, l)
                assert np.array_equal(b["A"][1], a["A"][1])
                assert not np.array_equal(b["A"][2], a["A"][2]), (w, l)
            if b["P"] is not None:
                assert all(np.array_equal(x, y) for x, y in zip(b["P"], a["P"]))
                A = oamg.galerkin(A, b["P"], oamg.transpose(b["P"], got[l + 1]["cf"].size))
    for s in (first, second, fresh, start):
        s.close()


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("known") / "known_pattern")
    lib = os.path.join(ROOT, "paper_1902_00095_gb300")
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off",
                        "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(lib, "csrc"), os.path.join(HERE, "known_pattern.cpp"),
                        os.path.join(lib, "libthermo.so"), "-Wl,-rpath," + lib,
                        "-L" + os.path.join(cuda, "lib64"), "-lcudart",
                        "-Wl,-rpath," + os.path.join(cuda, "lib64"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def test_products_on_known_patterns_of_every_row_class(harness):
    """C = A B anew on its pattern, rows of 1 to 3000 columns (the lane groups' three
    classes and the rows past them), against the sums in canonical order."""
    r = subprocess.run([harness], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
