"""Device arrays that a kernel uses where they lie give the bits of the same
call on host arrays; overlapping and unaligned ones go through copies and do
too."""
import ctypes as C

import numpy as np
import pytest

from synthetic import make_problem
from synthetic.recipes import perturbed_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


def at(buf, byte, values=None):
    """Address `byte` bytes into a device buffer, filled with `values` there."""
    if values is not None:
        raw = torch.from_numpy(np.ascontiguousarray(values).view(np.uint8).ravel().copy())
        buf[byte:byte + raw.numel()] = raw.cuda()
        torch.cuda.synchronize()
    return C.c_void_p(buf.data_ptr() + byte)


@pytest.mark.parametrize("shift", [0, 4, 1])
def test_spmv_on_device_arrays(shift):
    prob = make_problem("tiny", shape=(9, 7, 5), seed=2)
    s = thermo.Solver.from_problem(prob)
    s.assemble(*perturbed_state(prob, seed=3), prob["p_n"], prob["T_n"], prob["dt"])
    n = s.N
    x = np.random.default_rng(1).normal(size=(2, n))
    y = s.spmv(x[0], x[1])
    buf = torch.zeros(40 * n, dtype=torch.uint8, device="cuda")
    slot = lambda k: shift + 8 * n * k
    read = lambda k: buf[slot(k):slot(k) + 8 * n].cpu().numpy().copy().view(np.float64)
    # outputs apart, each in place of an input, swapped, and one in place of both
    for yp, yT in ((2, 3), (0, 1), (1, 0), (0, 3), (2, 1), (2, 2)):
        xs = [at(buf, slot(k), x[k]) for k in (0, 1)]
        assert thermo.load().tp_spmv(s._h, *xs, at(buf, slot(yp)), at(buf, slot(yT)), 1) == 0
        if yp != yT:
            assert np.array_equal(read(yp), y[0])
        assert np.array_equal(read(yT), y[1])
    s.close()


@pytest.mark.parametrize("shift", [0, 4, 2])
def test_training_batch_on_device_arrays(shift):
    rng = np.random.default_rng(5)
    B = 77
    Sd = rng.uniform(1, 2, B)
    arrays = [rng.normal(0, 1, (B, 24)).astype(np.float32), rng.integers(0, 7, B).astype(np.int32),
              -rng.uniform(0.05, 0.3, B), Sd, -rng.uniform(0.05, 0.3, B)]
    mlp = thermo.MLP(rng.normal(0, 0.1, thermo.NPARAM))
    loss, g = mlp.gradient(*arrays)
    buf = torch.zeros(B * 160 + 64, dtype=torch.uint8, device="cuda")
    ptrs, byte = [], shift
    for a in arrays:
        ptrs.append(at(buf, byte, a))
        byte += (a.nbytes + 7) // 8 * 8
    gd, ld = np.empty_like(g), C.c_double()
    assert thermo.load().tp_mlp_gradient(mlp._h, B, *ptrs, C.c_void_p(gd.ctypes.data),
                                         C.byref(ld), 1) == 0
    assert np.array_equal(gd, g) and ld.value == loss
