"""Calls on a device whose memory is nearly all taken give the results of the
same calls with memory to spare: what is kept for speed alone is left out or
given back."""
import ctypes as C

import numpy as np
import pytest

from synthetic import make_problem
from synthetic.recipes import perturbed_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


class Taken:
    """Takes device memory (in the process's context, past every pool) until at
    most `leave` bytes and 2 MiB are free."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        torch.cuda.synchronize()
        self.cuda = C.CDLL("libcuda.so.1")
        self.held = []
        for block in (1 << 33, 1 << 28, 1 << 21):
            while torch.cuda.mem_get_info()[0] >= self.leave + block:
                p = C.c_uint64()
                if self.cuda.cuMemAlloc_v2(C.byref(p), C.c_size_t(block)) != 0:
                    break
                self.held.append(p)
        return self

    def __exit__(self, *exc):
        for p in self.held:
            self.cuda.cuMemFree_v2(p)


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def solver(shape, seed=4):
    prob = make_problem("tiny", shape=shape, seed=seed)
    p, T = perturbed_state(prob, seed=seed + 1)
    s = thermo.Solver.from_problem(prob)
    s.assemble(p, T, prob["p_n"], prob["T_n"], prob["dt"])
    return s


# 800,000 cells: 45 MB a plane
def test_no_room_for_coupling_planes():
    shape = (100, 100, 80)
    ref = solver(shape)
    scales = ref.export_system()[4]
    ref.build(variant=1)
    x = ref.solve(rtol=1e-8)
    ref.close()
    s = solver(shape)
    for leave in (60 << 20, 16 << 20):  # one plane and not two; none
        with Taken(leave):
            assert np.array_equal(s.export_system()[4], scales)
    s.build(variant=1)
    y = s.solve(rtol=1e-8)
    assert y[2]["iters"] == x[2]["iters"] and np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
    s.close()


# 3,840 cells: the Krylov vectors lie in pool chunks of 4 to 16 MiB, the larger
# workspace's first vectors fit those that are there and its last ones do not
def test_krylov_workspace_that_could_not_grow():
    s = solver((16, 16, 15))
    s.build()
    x = s.solve(rtol=1e-8, restart=30)
    with Taken(0):
        with pytest.raises(thermo.ThermoError) as e:
            s.solve(rtol=1e-8, restart=100)
        assert e.value.status == thermo.TP_ENOMEM
    y = s.solve(rtol=1e-8, restart=30)
    assert y[2]["iters"] == x[2]["iters"] and np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
    s.close()


# 800,000 cells: 26 MB for the network's outputs, 45 MB for S~, 77 MB of features
def test_no_room_for_the_learned_work_arrays():
    s = solver((100, 100, 80))
    for leave in (85 << 20, 40 << 20):
        with Taken(leave):
            for _ in range(2):
                with pytest.raises(thermo.ThermoError) as e:
                    s.learned_features()
                assert e.value.status == thermo.TP_ENOMEM
    X = s.learned_features()
    s.close()
    r = solver((100, 100, 80))
    assert np.array_equal(X, r.learned_features())
    r.close()


# 131,072 cells: some 90 MB a lane. Room for a few lanes, for none, and again
# for all on the same context
def test_columns_with_room_for_few_lanes():
    s = solver((64, 64, 32))
    s.build()
    s.solve(rtol=1e-8)  # the context's own workspace
    cols = np.arange(0, s.N, 13001, dtype=np.int32)
    assert cols.size > 8
    one = [s.probe_schur_columns([c], rtol=1e-10) for c in cols]
    for leave in (16 << 20, 130 << 20, 300 << 20):
        with Taken(leave):
            entry, value, its, st = s.probe_schur_columns(cols, rtol=1e-10)
        assert st == 0 and its == sum(o[2] for o in one)
        assert np.array_equal(entry, np.concatenate([o[0] for o in one]))
        assert np.array_equal(value, np.concatenate([o[1] for o in one]))
    s.close()


# a larger Krylov workspace in 40 MB less than it takes: it fits only into what the
# lanes (131,072 cells), or the coupling planes (90 MB at 800,000 cells, with the
# graph recorded anew), give back
@pytest.mark.parametrize("shape", [(64, 64, 32), (100, 100, 80)])
def test_memory_kept_for_speed_is_given_back(shape):
    r = solver(shape)
    r.build()
    r.solve(rtol=1e-8, restart=30)
    f = free()
    x = r.solve(rtol=1e-8, restart=31)
    taken = f - free()
    r.close()
    s = solver(shape)
    s.build()
    s.solve(rtol=1e-8, restart=30)
    cols = [0, 1, 2]
    c0 = s.probe_schur_columns(cols, rtol=1e-10)
    with Taken(taken - (40 << 20)):
        y = s.solve(rtol=1e-8, restart=31)
    z = s.solve(rtol=1e-8, restart=31)
    c1 = s.probe_schur_columns(cols, rtol=1e-10)
    s.build()
    w = s.solve(rtol=1e-8, restart=31)
    s.close()
    assert np.array_equal(c0[0], c1[0]) and np.array_equal(c0[1], c1[1])
    for a in (y, z, w):
        assert a[2]["iters"] == x[2]["iters"]
        assert np.array_equal(a[0], x[0]) and np.array_equal(a[1], x[1])


# 800,000 cells, 90 MB of planes: a first build in 40 MB less than it takes
def test_build_in_the_memory_of_one_without_planes():
    r = solver((100, 100, 80))
    f = free()
    r.build()
    taken = f - free()
    x = r.solve(rtol=1e-8)
    r.close()
    s = solver((100, 100, 80))
    with Taken(taken - (40 << 20)):
        s.build()
    y = s.solve(rtol=1e-8)
    s.close()
    assert y[2]["iters"] == x[2]["iters"] and np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
