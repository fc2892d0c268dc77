"""The one-launch step of few hypercubes where the sum of d_h is not finite (the
allocation is kept) and with several outputs, against the separate calls."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_st", [300, 1500, 4000])  # 1, 2 and 4 blocks
@pytest.mark.parametrize("precision", [0, 1])
def test_nonfinite_sum_keeps_the_allocation(n_st, precision):
    # (J f)^2 overflows FP64: f ~ 1e300 over the whole box
    prob = inputs.Problem("inf", 1, inputs.GAUSS, inputs.gauss_blob([1e300], [10.0], [[0.5]]),
                          np.zeros(1), np.ones(1), n_g=40, n_ev=5 * n_st + 1, n_st=n_st, seed=n_st)
    a = vegasp.Integrator.from_problem(prob, precision=precision)
    b = vegasp.Integrator.from_problem(prob, precision=precision)
    n0, o0 = a.alloc()
    for it in range(3):
        a.step()
        b.iterate()
        b.adapt()
        for g in (a, b):
            n, off = g.alloc()
            assert np.array_equal(n, n0) and np.array_equal(off, o0)
            r = g.result(allow_nonfinite=True)
            assert r["status"] == vegasp.VP_ENONFINITE
            assert len(g.history()[0]) == it + 1
        assert np.array_equal(a.edges(), b.edges())
    a.close()
    b.close()


@pytest.mark.parametrize("n_st", [1023, 1025, 4096])
def test_several_outputs_equal_the_separate_calls(n_st):
    prob = inputs.Problem("m", 1, inputs.GAUSS, inputs.gauss_blob([1.0, 0.5], [0.2, 0.1],
                                                                  [[0.3], [0.7]]),
                          np.zeros(1), np.ones(1), n_g=60, n_ev=7 * n_st, n_st=n_st, seed=n_st)
    kw = dict(precision=vegasp.VP_FP64, out_mono=[(0, -1), (0, 0)])
    a = vegasp.Integrator.from_problem(prob, **kw)
    b = vegasp.Integrator.from_problem(prob, **kw)
    for _ in range(3):
        a.step()
        b.iterate()
        b.adapt()
    (ia, ca), (ib, cb) = a.history_multi(), b.history_multi()
    # (FP64 sums added in any order: the roundings of 3e4 terms, and of the
    # grids they lead to)
    assert np.allclose(ia, ib, rtol=1e-11, atol=0)
    s = np.sqrt(np.einsum("jkk,jll->jkl", cb, cb))
    assert np.all(np.abs(ca - cb) <= 1e-9 * s)
    a.close()
    b.close()
