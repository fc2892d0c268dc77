"""The launch shape of an FP32 part is a rule's, not a stopwatch's (its roundings
are in the exported sums): sampling a part measures nothing, and the sums are
those of the same part in another context to FP32 roundings, whatever that one
ran before."""
import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def problem(kind, dim, n_ev, mixed):
    rng = np.random.default_rng(dim)
    c = [rng.uniform(0.3, 0.7, dim)]
    blob = (inputs.gauss_blob([1.0], [0.3], c) if kind == inputs.GAUSS else
            inputs.expnorm_blob([1.0], [5.0], c))
    return inputs.Problem("p", dim, kind, blob, np.zeros(dim), np.ones(dim), n_g=1000, n_ev=n_ev,
                          mixed=mixed, seed=dim)


def sums(g, n_parts):
    buf = torch.empty(g.partials_size(), dtype=torch.float64, device="cuda")
    for p in range(n_parts):
        g.iterate_part(p, n_parts)
    g.export_partials(buf.data_ptr())
    torch.cuda.synchronize()
    return buf.cpu().numpy()


@pytest.mark.parametrize("kind,dim,n_ev,mixed", [
    (inputs.EXPNORM, 16, 250_001, True), (inputs.GAUSS, 2, 300_001, False),
    (inputs.GAUSS, 8, 600_001, False), (inputs.EXPNORM, 20, 400_001, False),
    (inputs.GAUSS, 11, 300_001, False), (inputs.GAUSS, 4, 100_001, False)])
def test_part_takes_the_rules_shape(kind, dim, n_ev, mixed):
    prob = problem(kind, dim, n_ev, mixed)
    a = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP32)
    before = a.tuning()
    x = sums(a, 3)
    assert a.tuning() == before  # (nothing measured: still the shape of a new context)
    b = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP32)
    b.iterate()  # measured, on the first iteration's allocation
    c = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP32)
    y = sums(c, 3)
    n, m = a.n_hc, dim * 1000
    assert np.array_equal(x[2 * n + m:], y[2 * n + m:])  # the counts
    # a bin's k nonnegative terms in FP32: each sum within k roundings of exact
    k = x[2 * n + m:]
    hx, hy = x[2 * n:2 * n + m], y[2 * n:2 * n + m]
    assert np.all(np.abs(hx - hy) <= 2.0 * (k + 8) * 2.0 ** -24 * np.maximum(hx, hy))
    for g in (a, b, c):
        g.close()
