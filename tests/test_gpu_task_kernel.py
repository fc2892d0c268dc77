"""The task kernel's loop per dimension and its histogram layouts (768 threads
up to 220 KB, else 256 and global adds) against the same integrals one by one."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


def member(kind, dim, n_g, i):
    rng = np.random.default_rng(100 * kind + dim)
    c = [rng.uniform(0.3, 0.7, dim) for _ in range(2)]
    blob = (inputs.gauss_blob([1.0, 0.5], [0.3, 0.2], c) if kind == inputs.GAUSS else
            inputs.ball_blob([0.6, 0.4], c) if kind == inputs.BALL else
            inputs.expnorm_blob([1.0, 0.5], [5.0, 8.0], c))
    return inputs.Problem("m", dim, kind, blob, np.zeros(dim), np.ones(dim), n_g=n_g,
                          n_ev=3001 + 97 * dim, seed=11, integral_id=i)


@pytest.mark.parametrize("kind", [inputs.GAUSS, inputs.BALL, inputs.EXPNORM])
@pytest.mark.parametrize("dims,n_g", [(range(1, 5), 50), (range(1, 9), 333), (range(1, 13), 1200),
                                      ((12, 11), 2000), (range(9, 25), 100)])
def test_batch_members_equal_single_integrals(kind, dims, n_g):
    probs = [member(kind, d, n_g, i) for i, d in enumerate(dims)]
    b = vegasp.Batch(probs, precision=vegasp.VP_FP32)
    b.run(2)
    for i, p in enumerate(probs):
        g = vegasp.Integrator.from_problem(p, precision=vegasp.VP_FP32)
        g.run(2)
        (ib, vb), (ig, vg) = b.history(i), g.history()
        # the same samples, summed in another order in single precision; the
        # second iteration's grid carries that order's roundings
        assert np.allclose(ib[0], ig[0], rtol=1e-5, atol=0)
        assert np.allclose(vb[0], vg[0], rtol=1e-4, atol=0)
        assert abs(ib[1] - ig[1]) <= 1e-3 * abs(ig[1]) + 0.1 * np.sqrt(vg[1])
        g.close()
    b.close()
