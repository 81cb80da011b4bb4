"""Training batches from host memory: through the pinned image, past its size and
after it, the gradient and the step of the same batch in device memory, bit for
bit."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


def batch(B):
    rng = np.random.default_rng(B)
    return [rng.normal(0, 1, (B, 24)).astype(np.float32), rng.integers(0, 7, B).astype(np.int32),
            -rng.uniform(0.05, 0.3, B), rng.uniform(1, 2, B), -rng.uniform(0.05, 0.3, B)]


# the image holds 3072 samples; the sizes grow, shrink and cross it both ways
@pytest.mark.parametrize("sizes", [(1, 17, 3071, 3072, 3073, 50, 20000, 3072, 1), (9000, 16)])
def test_host_batches_of_every_size(sizes):
    P = np.random.default_rng(1).normal(0, 0.1, thermo.NPARAM)
    host, dev = thermo.MLP(P), thermo.MLP(P)
    lib = thermo.load()
    for B in sizes:
        b = batch(B)
        d = [torch.from_numpy(a).cuda() for a in b]
        torch.cuda.synchronize()
        ptrs = [C.c_void_p(t.data_ptr()) for t in d]
        loss, g = host.gradient(*b)
        gd, ld = np.empty_like(g), C.c_double()
        assert lib.tp_mlp_gradient(dev._h, B, *ptrs, C.c_void_p(gd.ctypes.data), C.byref(ld), 1) == 0
        assert np.array_equal(g, gd) and loss == ld.value
        loss = host.train_step(*b, lr=1e-3)
        assert lib.tp_mlp_train_step(dev._h, B, *ptrs, 1e-3, C.byref(ld), 1) == 0
        assert loss == ld.value
        assert np.array_equal(host.params(), dev.params())
