"""One FP64 sample where its shortened steps could go wrong: k + u and the
division by the strata count at the ends of their ranges, 1/w^2 out of range."""
import math

import numpy as np
import pytest

import oracle
from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n_st,widths", [
    (1, 1, [0.1]), (1, 3, [0.2, 1e-160]), (1, 1 << 19, [0.05]), (1, (1 << 19) + 1, [0.05]),
    (1, 999_983, [1e152, 0.3]), (2, 725, [0.1, 1e-150, 2.0]), (3, 49, [1e150])])
def test_fp64_sample_equals_the_oracle(dim, n_st, widths):
    rng = np.random.default_rng(dim + n_st)
    K = len(widths)
    prob = inputs.Problem("p", dim, inputs.GAUSS,
                          inputs.gauss_blob([1.0] * K, widths,
                                            [rng.uniform(0.3, 0.7, dim) for _ in range(K)]),
                          np.zeros(dim), np.ones(dim), n_g=777, n_ev=2 * n_st ** dim + 2,
                          n_st=n_st, seed=int(rng.integers(1 << 40)))
    g = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP64)
    o = oracle.VegasPlus(dim=dim, lo=prob.lo, hi=prob.hi, n_g=prob.n_g, n_ev=prob.n_ev,
                         alpha=prob.alpha, beta=prob.beta, seed=prob.seed, kind=prob.kind,
                         prm=prob.prm, n_st=n_st)
    n = 400
    hs = rng.integers(0, g.n_hc, n).astype(np.uint64)
    hs[:2] = 0, g.n_hc - 1
    js = rng.integers(0, 50, n).astype(np.uint32)
    x, idx, jac, f = g.eval_samples(hs, js, 3)
    for k in range(n):
        xo, io, jo, fo = o.eval_sample(3, int(hs[k]), int(js[k]))
        assert np.array_equal(idx[k], io) and np.array_equal(x[k], xo) and jac[k] == jo
        # (exp of CUDA and of the host differ by an ulp or two)
        if fo > 0:
            assert f[k] > 0
            assert abs(math.log(f[k]) - math.log(fo)) <= 2e-14 * max(1.0, abs(math.log(fo)))
        else:
            assert f[k] == 0.0
    g.close()
