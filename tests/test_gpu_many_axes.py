"""The FP32 sampling loop's forms above 12 axes (indices packed or not, digits
kept or decoded; dimension-exact and guarded; one integral and several): the
histogram counts are those of the increments vp_eval_samples gives for every
sample of the iteration, exactly, and the hypercube sums those of its J f."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [13, 16, 17, 20, 23, 24])
@pytest.mark.parametrize("kind,peaks", [(inputs.GAUSS, 2), (inputs.EXPNORM, 3),
                                        (inputs.GAUSS, 12), (inputs.BALL, 1)])
@pytest.mark.parametrize("axes", [False, True])
def test_counts_and_sums(dim, kind, peaks, axes):
    rng = np.random.default_rng(dim + peaks)
    c = [rng.uniform(0.4, 0.6, dim) for _ in range(peaks)]
    blob = (inputs.gauss_blob([1.0] * peaks, [1.0] * peaks, c) if kind == inputs.GAUSS else
            inputs.ball_blob([1.3] * peaks, c) if kind == inputs.BALL else
            inputs.expnorm_blob([1.0] * peaks, [1.0] * peaks, c))
    strata = tuple(3 if mu in (0, dim - 1) else (2 if mu in (1, dim // 2) else 1)
                   for mu in range(dim))
    if axes and peaks > 8 and dim in (16, 20, 24):
        pytest.skip("strata per axis at an exact dimension: at most 8 peaks")
    prob = inputs.Problem("p", dim, kind, blob, np.zeros(dim), np.ones(dim), n_g=101, n_ev=3001,
                          n_st_axis=strata if axes else None, n_st=0 if axes else 1, seed=dim)
    g = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP32)
    n_h, _ = g.alloc()
    g.iterate()
    hsum, hcnt = g.hist()
    s1, s2 = g.moments()
    h = np.repeat(np.arange(g.n_hc, dtype=np.uint64), n_h)
    j = np.concatenate([np.arange(n, dtype=np.uint32) for n in n_h])
    _, idx, jac, f = g.eval_samples(h, j, 0)
    cnt = np.stack([np.bincount(idx[:, mu], minlength=101) for mu in range(dim)])
    assert np.array_equal(np.asarray(hcnt).reshape(dim, 101), cnt)
    # every J f is one FP32 number (its constants read from another memory: an
    # ulp or two of each of 3 dim operations), added compensated
    tol = 3 * dim * 2.0 ** -23
    ref = np.zeros(g.n_hc)
    np.add.at(ref, h.astype(int), jac * f)
    assert np.all(np.abs(s1 - ref) <= tol * ref + 1e-30)
    g.close()
