"""The step graph of an integral of few hypercubes (estimate, allocation and
offsets on one cluster) against the separate calls, around its block edges."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_st", [1, 2, 255, 257, 1023, 1024, 1025, 2048, 2049, 3073, 4095, 4096,
                                  4097])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("plus2", [False, True])
def test_step_equals_iterate_and_adapt(n_st, precision, plus2):
    prob = inputs.Problem("p", 1, inputs.GAUSS, inputs.gauss_blob([1.0, 0.5], [0.1, 0.03],
                                                                  [[0.3], [0.71]]),
                          np.zeros(1), np.ones(1), n_g=40, n_ev=max(20 * n_st, 500), n_st=n_st,
                          plus2=plus2, seed=n_st)
    a = vegasp.Integrator.from_problem(prob, precision=precision)
    b = vegasp.Integrator.from_problem(prob, precision=precision)
    # (FP32: the grid's FP32 sums, added in any order, part the runs after one step)
    for it in range(1 if precision else 3):
        a.step()
        b.iterate()
        b.adapt()
        na, oa = a.alloc()
        nb, ob = b.alloc()
        # (the reductions' order differs between runs by roundings, which move
        # an n_h only where a quotient falls on an integer)
        assert np.count_nonzero(na != nb) <= 1 and np.abs(na.astype(int) - nb.astype(int)).max() <= 1
        assert np.array_equal(oa, np.concatenate([[0], np.cumsum(na.astype(np.uint64))]))
        ia, va = a.history()
        ib, vb = b.history()
        assert np.allclose(ia, ib, rtol=1e-6 if precision else 1e-12, atol=0)
        assert np.allclose(va, vb, rtol=1e-5 if precision else 1e-10, atol=0)
    a.close()
    b.close()
