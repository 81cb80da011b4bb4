"""Exact Schur columns solved side by side are the columns solved one at a time
(the same operations per column, so the same bits), for more columns than
lanes, with every hierarchy storage and smoother, and after a rebuild."""
import numpy as np
import pytest

from synthetic import make_problem
from synthetic.recipes import perturbed_state

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


@pytest.mark.parametrize("shape,opts", [((12, 11, 7), {}), ((12, 11, 7), dict(precision=1)),
                                        ((9, 1, 13), dict(precision=2)),
                                        ((12, 11, 7), dict(smoother=1)),
                                        ((12, 11, 7), dict(max_levels=1, coarse_size=2048)),
                                        ((12, 11, 7), dict(use_graphs=0)),
                                        ((12, 11, 7), dict(tail_rows=400))])
def test_columns_side_by_side_equal_columns_one_by_one(shape, opts):
    prob = make_problem("tiny", shape=shape, seed=4)
    p, T = perturbed_state(prob, seed=5)
    s = thermo.Solver.from_problem(prob)
    n = s.N
    cols = np.concatenate([[0, n - 1, n // 2, n // 2], np.arange(1, 16)]).astype(np.int32)
    for state in ((p, T), (prob["p_k"] + 1.0e3, prob["T_k"])):  # a second build on the lanes
        s.assemble(*state, prob["p_n"], prob["T_n"], prob["dt"])
        s.build(**opts)
        entry, value, its, st = s.probe_schur_columns(cols, rtol=1e-10)
        assert st == 0
        one = [s.probe_schur_columns([c], rtol=1e-10) for c in cols]
        assert np.array_equal(entry, np.concatenate([o[0] for o in one]))
        assert np.array_equal(value, np.concatenate([o[1] for o in one]))
        assert its == sum(o[2] for o in one)
    with pytest.raises(thermo.ThermoError) as e:
        s.probe_schur_columns([0, 1, n], rtol=1e-10)
    assert e.value.status == thermo.TP_EINVAL
    assert s.probe_schur_columns(np.zeros(0, np.int32))[2] == 0
    s.close()
