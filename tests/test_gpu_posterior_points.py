"""The FP32 posterior's points for every count of coefficients around its groups
of four (1, 2 and 3 with the value, then 4 at a time), dimension-exact and
guarded, fewer points than weights among them: f at the sample's own x against
the formula in 64 bits on the constants as the kernel holds them (FP32)."""
import math

import numpy as np
import pytest

from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def log2_f(prm, x):
    """log2 f, and how far FP32 arithmetic may be from it: every rounding u of
    its operand, the approximate exponentials and logarithms 2^-21, each
    exponent's error in proportion to its term's share of the mixture."""
    n, P, G = (int(v) for v in prm[:3])
    sy, pw, ref = prm[3:6]
    y = prm[6:6 + n].astype(np.float32).astype(float)
    A = prm[6 + n:].reshape(n, P).astype(np.float32).astype(float)
    L2E = 1.0 / math.log(2.0)
    kN, kW = L2E / (2.0 * sy * sy), L2E / (200.0 * sy * sy)
    lN, lW = math.log2(1.0 / (math.sqrt(2.0 * math.pi) * sy)), math.log2(1.0 / (math.sqrt(2.0 * math.pi) * 10.0 * sy))
    acc, err, top = 0.0, 0.0, 0.0
    for i in range(n):
        w = x[P + i % G]
        r = float(y[i] - A[i] @ x[:P])
        dr = U * (P + 2) * (abs(y[i]) + float(np.abs(A[i]) @ np.abs(x[:P])))
        aN, aW = lN + math.log2(1.0 - w) - kN * r * r, lW + math.log2(w) - kW * r * r
        t = float(np.logaddexp2(aN, aW))
        for k, a, c in ((kN, aN, lN), (kW, aW, lW)):
            share = 2.0 ** (a - t)
            err += share * (2.0 * k * abs(r) * dr + k * dr * dr + 6.0 * U * k * r * r +
                            8.0 * U * (abs(c) + 8.0) + 2.0 ** -20)
        err += 2.0 ** -20
        acc += t
        top = max(top, abs(acc))
    prior, lref = float(np.sum(x[:P] ** 2)) * L2E / (2.0 * pw * pw), ref * L2E
    err += U * ((n + 4) * top + (P + 6) * prior + 6.0 * abs(lref) + 8.0) + 2.0 ** -20
    return acc - prior - lref, 2.0 * err


@pytest.mark.parametrize("dim,par", [(2, 1), (3, 2), (4, 3), (4, 2), (5, 3), (6, 4), (8, 5), (8, 6),
                                     (8, 7), (9, 8), (11, 7), (12, 11), (14, 3), (16, 12),
                                     (20, 19), (21, 20), (22, 2), (24, 23)])
@pytest.mark.parametrize("n", [1, 3, 50])
def test_points(dim, par, n):
    rng = np.random.default_rng(100 * dim + par + n)
    G = dim - par
    A = rng.uniform(-1.0, 1.0, (n, par))
    y = A @ rng.normal(0.0, 0.3, par) + rng.normal(0.0, 0.3, n)
    prm = np.concatenate([[n, par, G, 0.5, 1.0, 0.0], y, A.ravel()])
    lo, hi = np.concatenate([np.full(par, -1.0), np.full(G, 0.02)]), np.concatenate([np.full(par, 1.0), np.full(G, 0.98)])
    prob = inputs.Problem("post", dim, inputs.POSTERIOR, prm, lo, hi, n_g=50, n_ev=2000, seed=5)
    g = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP32)
    hs = rng.integers(0, g.n_hc, 100).astype(np.uint64)
    js = rng.integers(0, 50, 100).astype(np.uint32)
    x, _, _, f = g.eval_samples(hs, js, 2)
    g.close()
    for k in range(100):
        want, tol = log2_f(prm, x[k])
        assert abs(math.log2(f[k]) - want) <= tol, (k, f[k], want, tol)
