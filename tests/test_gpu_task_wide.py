"""The task kernel's two CTAs (256 threads, two per SM; 768, one, for large sets
of FP32 peaks) on both sides of the lines between them, with the same strata on
every axis and strata that differ, against the same integrals one by one."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu


def member(kind, dim, n_g, n_ev, mixed, i):
    rng = np.random.default_rng(100 * kind + dim)
    c = [rng.uniform(0.3, 0.7, dim) for _ in range(2)]
    blob = (inputs.gauss_blob([1.0, 0.5], [0.3, 0.2], c) if kind == inputs.GAUSS else
            inputs.ball_blob([0.6, 0.4], c) if kind == inputs.BALL else
            inputs.expnorm_blob([1.0, 0.5], [5.0, 8.0], c))
    return inputs.Problem("m", dim, kind, blob, np.zeros(dim), np.ones(dim), n_g=n_g,
                          n_ev=n_ev + 97 * dim, seed=11, integral_id=i, mixed=mixed)


@pytest.mark.parametrize("kind,dims,n_g,n_ev,mixed", [
    (inputs.GAUSS, range(1, 13), 500, 300_000, False),      # wide, every dimension's loop
    (inputs.BALL, range(1, 13), 250, 300_000, False),
    (inputs.EXPNORM, range(1, 13), 1200, 150_000, False),   # wide only holds the histograms
    (inputs.GAUSS, (8, 8, 8), 333, 800_000, False),         # wide, dimension-exact
    (inputs.BALL, (4, 4, 4, 4), 333, 500_000, False),
    (inputs.EXPNORM, (4, 3, 4, 3, 3), 77, 400_000, False),
    (inputs.GAUSS, (3, 4, 3), 333, 700_000, False),         # three of few axes: 256 threads
    (inputs.BALL, (2, 1, 2, 5), 333, 600_000, False),       # most samples on two axes
    (inputs.EXPNORM, (6, 7), 333, 400_000, False),          # too few samples
    (inputs.GAUSS, (12, 11), 2000, 1_000_000, False),       # histograms in global memory
    (inputs.EXPNORM, (5, 7, 10, 12), 400, 1_200_000, True),  # wide, strata per axis
    (inputs.GAUSS, (5, 7, 10, 12), 400, 300_000, True)])
def test_batch_members_equal_single_integrals(kind, dims, n_g, n_ev, mixed):
    probs = [member(kind, d, n_g, n_ev, mixed, i) for i, d in enumerate(dims)]
    b = vegasp.Batch(probs, precision=vegasp.VP_FP32)
    b.run(1)
    for i, p in enumerate(probs):
        g = vegasp.Integrator.from_problem(p, precision=vegasp.VP_FP32)
        n_h = g.alloc()[0].astype(float)
        g.run(1)
        s1, s2 = g.moments()
        (ib, vb), (ig, vg) = b.history(i), g.history()
        # the same samples, each J f to an ulp or two of 3 D operations (their
        # constants come from another memory); the sums are compensated.  The
        # variances take the difference of two such numbers per hypercube
        e = 3 * p.dim * 2.0 ** -23
        assert abs(ib[0] - ig[0]) <= e * abs(ig[0])
        second = np.sum(s2 / n_h / (n_h - 1.0)) / g.n_hc ** 2
        assert abs(vb[0] - vg[0]) <= 4.0 * e * second
        g.close()
    b.close()
