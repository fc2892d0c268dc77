"""The FP64 posterior where its product form could part from the sum of
logarithms: noise widths whose squared reciprocals leave the range of the
corrected product, residuals whose squares do, mixture terms that are
subnormal, zero or negative, products far outside the doubles, a reference
logarithm beyond the range of one exponential."""
import math

import numpy as np
import pytest

import oracle
from paper_2009_05112_gb300 import inputs

vegasp = pytest.importorskip("paper_2009_05112_gb300.vegasp")
pytestmark = pytest.mark.gpu

EPS, TINY = 2.0 ** -53, 2.0 ** -1074


def bound(prm, x):
    """How far log f may be from the same formula's on another IEEE machine:
    the roundings of both, each exponent's error in proportion to its term's
    share of the mixture, the subnormal numbers' by their absolute spacing."""
    n, P, G = (int(v) for v in prm[:3])
    sy, pw, ref = prm[3:6]
    y, A = prm[6:6 + n], prm[6 + n:].reshape(n, P)
    err, logl, worst = 0.0, 0.0, 0.0
    for i in range(n):
        w = x[P + i % G]
        r = float(y[i] - A[i] @ x[:P])
        dr = (P + 2) * EPS * (abs(y[i]) + float(np.abs(A[i]) @ np.abs(x[:P])))
        an, aw = (r / sy) ** 2 / 2.0, (r / sy) ** 2 / 200.0
        ln = math.log1p(-w) - math.log(math.sqrt(2 * math.pi) * sy) - an
        lw = math.log(w) - math.log(math.sqrt(2 * math.pi) * 10.0 * sy) - aw
        lt = float(np.logaddexp(ln, lw))
        for a, l in ((an, ln), (aw, lw)):
            share = math.exp(l - lt)
            err += share * (EPS * (8.0 * a + 16.0) + (2.0 * a * dr / abs(r) if r else 0.0))
            err += share * min(1.0, 3.0 * TINY / max(math.exp(-min(a, 744.0)), TINY))
        err += min(1.0, 2.0 * TINY / max(math.exp(min(max(lt, -744.0), 700.0)), TINY))
        logl += lt
        worst = max(worst, abs(logl))
    lp = float(np.sum(x[:P] ** 2)) / (2.0 * pw * pw)
    err += EPS * ((n + 8) * worst + (P + 8) * lp + 8.0 * abs(ref) + 16.0)
    f = logl - lp - ref
    return 2.0 * (err + 3.0 * TINY / max(math.exp(min(max(f, -744.0), 700.0)), TINY)), f


def blob(n, P, G, sy, ref, y, A=None, pw=1.0):
    A = np.zeros((n, P)) if A is None else A
    return np.concatenate([[n, P, G, sy, pw, ref], np.broadcast_to(y, (n,)), np.ravel(A)])


CASES = {
    # fast 0 for a wide noise: residuals whose squares pass 2^664 but whose
    # exponents are -50 and -2, and one beyond the square root of the largest double
    "wide noise": blob(2, 2, 1, 1e100, -460.0, [1e101, 3e100]),
    "wide noise, three points": blob(3, 1, 2, 2.0 ** 332, -690.5, [2.0 ** 333, -2.0 ** 334, 1e98]),
    "wide noise, square of the residual infinite": blob(1, 1, 1, 1e100, -230.0, [1e160]),
    # fast 0 for a narrow one (2 sy^2 below 2^-400), residuals of its size
    "narrow noise": blob(2, 2, 1, 2.0 ** -220, 300.0, [2.0 ** -219, 3 * 2.0 ** -221]),
    # the edges of fast
    "last reciprocal": blob(1, 1, 1, 2.0 ** 196, -130.0, [2.0 ** 198]),
    "first division": blob(1, 1, 1, 2.0 ** 197, -130.0, [2.0 ** 199]),
    # fast 1, r^2 beyond 2^664 and beyond the doubles: both exponentials zero
    "far residual": blob(2, 1, 1, 0.1, 0.0, [2.0 ** 333, 0.3]),
    "infinite square": blob(2, 1, 1, 0.1, 0.0, [1e200, 0.3]),
    # a subnormal mixture term, alone and brought back by the reference
    "subnormal term": blob(2, 1, 1, 1.0, -715.0, [math.sqrt(200.0 * 716.0), 0.5]),
    "subnormal exponential": blob(2, 1, 1, 1e-30, -600.0, [1e-30 * math.sqrt(200.0 * 720.0), 0.0]),
    # products far outside the doubles, brought back by the reference
    "large product": blob(60, 1, 1, 1e-10, 690.0 + 600.0, [0.0]),
    "large product, |z| below 700": blob(45, 1, 1, 1e-7, 600.0, [0.0]),
    "small product, |z| below 700": blob(45, 1, 1, 1e6, -640.0, [0.0]),
    "small product": blob(60, 2, 3, 1e9, -1290.0, [0.0]),
    # f itself outside: infinite, zero, subnormal
    "infinite": blob(60, 1, 1, 1e-10, 300.0, [0.0]),
    "zero": blob(60, 1, 1, 1e10, -300.0, [0.0]),
    "subnormal": blob(30, 1, 1, 1e10, 0.0, [0.0] * 30),
    # |z| at the limit of one exponential, both sides, through the prior too
    "z just below": blob(20, 1, 1, 1e-14, 699.5, [0.0], pw=1e3),
    "z just above": blob(20, 1, 1, 1e-14, 700.5, [0.0], pw=1e3),
    "z just below, negative reference": blob(20, 1, 1, 1e15, -699.5, [0.0], pw=1e3),
    "prior beyond": blob(20, 1, 1, 1e-17, 0.0, [0.0], pw=0.02),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_posterior_equals_the_oracle(name):
    prm = np.asarray(CASES[name], float)
    P, G = int(prm[1]), int(prm[2])
    D = P + G
    lo, hi = np.concatenate([np.full(P, -1.0), np.full(G, 0.05)]), np.concatenate([np.full(P, 1.0), np.full(G, 0.95)])
    prob = inputs.Problem("post", D, inputs.POSTERIOR, prm, lo, hi, n_g=50, n_ev=1000, seed=5)
    g = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP64)
    o = oracle.VegasPlus(dim=D, lo=lo, hi=hi, n_g=50, n_ev=1000, alpha=prob.alpha, beta=prob.beta,
                         seed=5, kind=prob.kind, prm=prm)
    rng = np.random.default_rng(1)
    n = 200
    hs = rng.integers(0, g.n_hc, n).astype(np.uint64)
    js = rng.integers(0, 50, n).astype(np.uint32)
    x, idx, jac, f = g.eval_samples(hs, js, 2)
    g.close()
    for k in range(n):
        xo, _, _, fo = o.eval_sample(2, int(hs[k]), int(js[k]))
        assert np.array_equal(x[k], xo)
        if not 0.0 < fo < math.inf:
            assert f[k] == fo
            continue
        assert 0.0 < f[k] < math.inf
        tol, _ = bound(prm, xo)
        assert abs(math.log(f[k]) - math.log(fo)) <= tol + 4.0 * EPS * abs(math.log(fo)), (f[k], fo)


def test_negative_mixture_is_not_a_number():
    """Weights outside [0, 1] (the box is the caller's): a negative term has no
    logarithm, two of them neither."""
    for pts in (1, 2):
        prm = blob(pts, 1, 1, 1.0, 0.0, [0.0] * pts)
        lo, hi = np.array([-1.0, 1.5]), np.array([1.0, 2.5])
        prob = inputs.Problem("post", 2, inputs.POSTERIOR, prm, lo, hi, n_g=50, n_ev=1000, seed=5)
        g = vegasp.Integrator.from_problem(prob, precision=vegasp.VP_FP64)
        o = oracle.VegasPlus(dim=2, lo=lo, hi=hi, n_g=50, n_ev=1000, alpha=prob.alpha,
                             beta=prob.beta, seed=5, kind=prob.kind, prm=prm)
        hs, js = np.arange(100, dtype=np.uint64) % g.n_hc, np.arange(100, dtype=np.uint32) % 7
        _, _, _, f = g.eval_samples(hs, js, 2)
        g.close()
        ref = np.array([o.eval_sample(2, int(h), int(j))[3] for h, j in zip(hs, js)])
        assert np.array_equal(np.isnan(f), np.isnan(ref)) and np.isnan(ref).any()
