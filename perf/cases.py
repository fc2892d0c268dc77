"""The work this library is measured on, through its public entry points.

Every case is a dict of plain values.  ``call`` says which use it stands for:

``job``         one integral from nothing to its result: create a context, run
                ``n_it`` adapting iterations, read the result, the history and
                the grid, close (what a program does that integrates a function
                once, the paper's way).
``production``  the measurement phase (a trained map, frozen as §2.5 and §3.2
                do, while the allocation keeps adapting): ``n_it`` steps of a
                context the program holds, their estimates streamed back.
``parts``       one integral sampled in ``parts`` ranges as several devices
                would: every range, then the partial sums out to a device
                buffer and back, the estimate and the reallocation.
``batch``       many independent integrals from nothing to their results.
``serve``       a queue of integration requests of mixed sizes, until all are
                answered.
``alloc``       the reallocation alone on the caller's device buffers.

Sizes are those of the repository's own workloads (inputs.py, bench.py, the
tests) or drawn from the ranges between them.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2009_05112_gb300 import inputs, vegasp

FAMILY = {"gauss": inputs.GAUSS, "ball": inputs.BALL, "exp": inputs.EXPNORM,
          "posterior": inputs.POSTERIOR}
PREC = {"fp64": vegasp.VP_FP64, "fp32": vegasp.VP_FP32}


def listed():
    return [
        # The smallest whole job: 3 peaks in 4-D, 1e4 samples per iteration,
        # the library's default precision.  Creation, launches and latency.
        dict(name="job_d4_fp64_1e4", call="job", family="gauss", dim=4, peaks=3, n_ev=10_000,
             n_g=1000, precision="fp64", n_it=10),
        # The 8-D four peaks as a whole adapting job at 1e6 samples, FP32 path.
        dict(name="job_d8_fp32_1e6", call="job", family="gauss", dim=8, peaks=4, n_ev=1_000_000,
             n_g=1000, precision="fp32", n_it=20),
        # The Bayesian fit of App. B with its means and second moments: eight
        # outputs and their covariance from the same samples (FP64 only).
        dict(name="job_bayes_d3_fp64_1e5", call="job", family="posterior", dim=3, points=50,
             n_ev=100_000, n_g=1000, precision="fp64", n_it=15, outputs=8),
        # The smallest steps in production: the 3-parameter posterior at 1e4.
        dict(name="steps_post_d3_fp32_1e4", call="production", family="posterior", dim=3,
             points=50, n_ev=10_000, n_g=1000, precision="fp32", n_it=16),
        # A ragged middle: odd dimension, odd counts, the exponential peaks.
        dict(name="steps_exp_d7_fp32_3e5", call="production", family="exp", dim=7, peaks=3,
             n_ev=300_007, n_g=777, precision="fp32", n_it=12),
        # The four peaks at 1e6 on the FP64 path (the default precision).
        dict(name="steps_d8_fp64_1e6", call="production", family="gauss", dim=8, peaks=4,
             n_ev=1_000_000, n_g=1000, precision="fp64", n_it=4),
        # The 20-D ball at 1e7 (2^20 hypercubes), the benchmark's default line.
        dict(name="steps_ball_d20_fp32_1e7", call="production", family="ball", dim=20, peaks=1,
             n_ev=10_000_000, n_g=1000, precision="fp32", n_it=4),
        # The largest single integral: 1e8 samples, 16.7 million hypercubes.
        dict(name="steps_d8_fp32_1e8", call="production", family="gauss", dim=8, peaks=4,
             n_ev=100_000_000, n_g=1000, precision="fp32", n_it=2),
        # Sharded sampling with the mixed strata of §3.2: exp(-50|x|) in 16-D,
        # sums weighted by 1/n_h, in four ranges; every sum comes back.
        dict(name="parts_mixed_d16_fp32_2.5e5", call="parts", family="exp", dim=16, peaks=1,
             n_ev=250_000, n_g=1000, precision="fp32", parts=4, mixed=True, weighted=True),
        # 512 uneven integrals iterated together, from nothing to the results.
        dict(name="batch_mix_512_fp32", call="batch", members=512, n_ev_lo=10_000,
             n_ev_hi=1_000_000, dim_lo=2, dim_hi=12, n_g=500, precision="fp32", n_it=15),
        # Posterior requests, 70% with 3 parameters and 30% with 21, served
        # together (24 of each family's iterations, whatever the accuracy).
        dict(name="serve_posteriors_256", call="serve", requests=256, share_d21=0.3,
             n_ev_d3=10_000, n_ev_d21=30_000, n_g=1000, precision="fp32", n_it=24),
        # The reallocation on device buffers: 6^8 hypercubes.
        dict(name="alloc_static_1.7M", call="alloc", n_hc=1_679_616, n_ev=10_000_000,
             plus2=False),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    call = rng.choice(["job"] * 3 + ["production"] * 7 + ["parts"] * 2 + ["batch"] * 2 +
                      ["serve"] * 2 + ["alloc"] * 2)
    if call == "alloc":
        n_hc = _log_uniform(rng, 1_000, 4_194_304)
        return dict(call=call, n_hc=n_hc, n_ev=_log_uniform(rng, 4 * n_hc, 100_000_000),
                    plus2=rng.random() < 0.25)
    precision = "fp32" if call in ("batch", "serve") or rng.random() < 0.65 else "fp64"
    if call == "batch":
        return dict(call=call, members=_log_uniform(rng, 16, 512), n_ev_lo=10_000,
                    n_ev_hi=rng.choice([100_000, 300_000, 1_000_000]), dim_lo=2,
                    dim_hi=rng.randint(4, 12), n_g=rng.choice([250, 500, 777]),
                    precision=precision, n_it=rng.randint(5, 15))
    if call == "serve":
        return dict(call=call, requests=_log_uniform(rng, 16, 256),
                    share_d21=round(rng.uniform(0.0, 0.3), 3), n_ev_d3=10_000, n_ev_d21=30_000,
                    n_g=rng.choice([500, 1000]), precision=precision, n_it=rng.randint(8, 24))
    family = rng.choice(["gauss", "gauss", "ball", "exp", "posterior"])
    single_job = call == "job" and precision == "fp32"
    if single_job:
        family = rng.choice(["gauss", "ball", "exp"])
    case = dict(call=call, family=family, n_g=rng.choice([250, 500, 777, 1000, 1000]),
                precision=precision)
    top = {"job": 1_000_000, "production": 30_000_000, "parts": 3_000_000}[call]
    if precision == "fp64":
        top = min(top, 2_000_000)
    if family == "posterior":
        case.update(dim=rng.choice([3, 3, 21]), points=rng.randint(20, 60))
        top = min(top, 1_000_000)
    else:
        # (an untrained run at these sizes only finds its peaks in a few dimensions)
        case.update(dim=rng.randint(4 if single_job else 2, 8 if call == "job" else 20),
                    peaks=rng.randint(1, 4))
    case["n_ev"] = _log_uniform(rng, 100_000 if single_job else 10_000, top) | 1
    if call == "parts":
        case.update(parts=rng.randint(1, 8), weighted=rng.random() < 0.3,
                    mixed=case["dim"] > 9 and rng.random() < 0.5)
    else:
        case["n_it"] = rng.randint(5, 15) if call == "job" else max(
            1, min(16, 4_000_000 // case["n_ev"]))
        if call == "job" and family == "posterior" and precision == "fp64":
            case["outputs"] = rng.choice([1, 3, 8])
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _problem(case, seed):
    """The integral of a case: box, integrand blob, settings."""
    rng = np.random.default_rng(seed)
    dim, family = case["dim"], case["family"]
    kw = dict(n_ev=case["n_ev"], n_g=case["n_g"], mixed=bool(case.get("mixed", False)),
              d_weighted=bool(case.get("weighted", False)))
    if family == "posterior":
        p = inputs.posterior(dim=dim, n_pts=case["points"], seed=int(rng.integers(1 << 31)))
        return inputs.Problem("post", dim, inputs.POSTERIOR, p.prm, p.lo, p.hi,
                              seed=int(rng.integers(1 << 62)), **kw)
    K = case["peaks"]
    amps = rng.uniform(0.5, 2.0, size=K)
    if family == "gauss":  # peaks on the diagonal, as in four_peaks_d8
        cs = [np.full(dim, (k + 1.0) / (K + 1.0)) for k in range(K)]
        prm = inputs.gauss_blob(amps, [0.1] * K, cs)
    elif family == "ball":  # one of half the box's width, others smaller around it
        cs = [np.full(dim, 0.5)] + [rng.uniform(0.4, 0.6, size=dim) for _ in range(K - 1)]
        prm = inputs.ball_blob([0.5] + [0.3] * (K - 1), cs, amps=amps)
    else:
        cs = ([np.zeros(dim)] if K == 1 else
              [np.full(dim, c) + rng.uniform(-0.03, 0.03, size=dim)
               for c in (0.23, 0.39, 0.74, 0.55)[:K]])
        prm = inputs.expnorm_blob(amps, [50.0] * K, cs)
    return inputs.Problem(family, dim, FAMILY[family], prm, np.zeros(dim), np.ones(dim),
                          seed=int(rng.integers(1 << 62)), **kw)


def _trained_grid(prob):
    """A map as training leaves it: on every axis the edges of equal shares of
    the root of the integrand's squared marginal, over a flat floor."""
    D, G = prob.dim, prob.n_g
    lo, hi = np.asarray(prob.lo, float), np.asarray(prob.hi, float)
    centre, spread, weight = [], [], []  # per component: centre [D], width [D], weight
    if prob.kind == inputs.POSTERIOR:
        n, P = int(prob.prm[0]), int(prob.prm[1])
        sy, y = prob.prm[3], prob.prm[6:6 + n]
        A = prob.prm[6 + n:].reshape(n, P)
        keep = np.ones(n, bool)
        for _ in range(5):  # least squares without the outliers
            c, *_ = np.linalg.lstsq(A[keep], y[keep], rcond=None)
            keep = np.abs(y - A @ c) < 4.0 * sy
        s = sy * np.sqrt(np.diag(np.linalg.inv(A[keep].T @ A[keep])))
        m = np.concatenate([c, np.full(D - P, 0.15)])
        centre, spread, weight = [m], [np.concatenate([2.0 * s, np.full(D - P, 0.2)])], [1.0]
    else:
        for row in prob.prm[1:].reshape(int(prob.prm[0]), 2 + D):
            centre.append(row[2:])
            w = row[1] if prob.kind != inputs.EXPNORM else math.sqrt(D) / row[1]
            spread.append(np.full(D, w))
            weight.append(row[0])
    edges = np.empty((D, G + 1))
    for mu in range(D):
        x = np.linspace(lo[mu], hi[mu], 8 * G + 1)
        p = np.full(x.size, 0.0)
        for c, s, a in zip(centre, spread, weight):
            z = (x - c[mu]) / s[mu]
            if prob.kind == inputs.BALL:
                p += a * np.maximum(1.0 - z * z, 0.0) ** ((D - 1) / 4.0)
            elif prob.kind == inputs.EXPNORM:
                p += a * np.exp(-np.abs(z))
            else:
                p += a * np.exp(-z * z)
        p = p / p.max() + 0.01
        cum = np.concatenate([[0.0], np.cumsum(0.5 * (p[1:] + p[:-1]))])
        edges[mu] = np.interp(np.linspace(0.0, cum[-1], G + 1), cum, x)
        edges[mu, 0], edges[mu, -1] = lo[mu], hi[mu]
    return edges


def _monomials(outputs):
    """The first `outputs` - 1 of the means and second moments of the
    3-parameter fit: <x0>, <x1>, <w>, <x0 x0>, <x0 x1>, <x1 x1>, <w w>."""
    return [(0, -1), (1, -1), (2, -1), (0, 0), (0, 1), (1, 1), (2, 2)][:outputs - 1]


def _members(case, seed):
    """Uneven Gaussian-peak integrals, as in inputs.batch_mix."""
    rng = np.random.default_rng(seed)
    out = []
    for b in range(case["members"]):
        dim = int(rng.integers(case["dim_lo"], case["dim_hi"] + 1))
        n_ev = int(round(math.exp(rng.uniform(math.log(case["n_ev_lo"]),
                                              math.log(case["n_ev_hi"])))))
        k = int(rng.integers(1, 5))
        cs = [rng.uniform(0.1, 0.9, size=dim) for _ in range(k)]
        out.append(inputs.Problem("m%d" % b, dim, inputs.GAUSS,
                                  inputs.gauss_blob([1.0] * k, rng.uniform(0.05, 0.2, size=k), cs),
                                  np.zeros(dim), np.ones(dim), n_g=case["n_g"], n_ev=n_ev,
                                  seed=seed, integral_id=b))
    return out


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["requests"]):
        dim = 21 if rng.random() < case["share_d21"] else 3
        n_ev = case["n_ev_d21"] if dim == 21 else case["n_ev_d3"]
        p = inputs.posterior(dim=dim, seed=int(rng.integers(1 << 31)))
        out.append(inputs.Problem("r%d" % i, dim, inputs.POSTERIOR, p.prm, p.lo, p.hi,
                                  n_g=case["n_g"], n_ev=n_ev, seed=int(rng.integers(1 << 62)),
                                  integral_id=i))
    return out


def _alloc_d(case, seed):
    """d_h as sharp peaks leave them: log-normal over many decades, a fifth zero."""
    rng = np.random.default_rng(seed)
    d = np.exp(rng.normal(0.0, 3.0, size=case["n_hc"]))
    d[rng.random(case["n_hc"]) < 0.2] = 0.0
    return d


def prepare(case, seed):
    torch.cuda.current_device()
    call = case["call"]
    st = dict(case=case)
    if call == "alloc":
        st["d"] = torch.from_numpy(_alloc_d(case, seed)).cuda()
        st["n"] = torch.empty(case["n_hc"], dtype=torch.int32, device="cuda")
        st["off"] = torch.empty(case["n_hc"] + 1, dtype=torch.int64, device="cuda")
    elif call == "batch":
        st["members"] = _members(case, seed)
    elif call == "serve":
        st["requests"] = _requests(case, seed)
        st["server"] = vegasp.Server()
    else:
        st["prob"] = prob = _problem(case, seed)
        if call == "job":
            if case.get("outputs", 1) > 1:
                st["mono"] = _monomials(case["outputs"])
        else:
            g = vegasp.Integrator.from_problem(prob, precision=PREC[case["precision"]])
            g.set_edges(_trained_grid(prob))
            g.set_damping(0.0, prob.beta)
            st["g"] = g
            if call == "parts":
                st["buf"] = torch.empty(g.partials_size(), dtype=torch.float64, device="cuda")
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _run_job(st):
    case = st["case"]
    g = vegasp.Integrator.from_problem(st["prob"], precision=PREC[case["precision"]],
                                       out_mono=st.get("mono"))
    g.run(case["n_it"])
    i, v = g.history()
    out = dict(i=i, sdev=np.sqrt(v), edges=g.edges())
    if "mono" in st:
        out["i_multi"], out["cov_multi"] = g.history_multi()
    if case["precision"] == "fp64":
        out["mean"] = g.result(discard=2)["mean"]
        out["n_h"] = g.alloc()[0].astype(np.int64)
    else:  # single precision samples
        out = {k: x.astype(np.float32) for k, x in out.items()}
    g.close()
    return out


def _run_production(st):
    g = st["g"]
    got = [g.step_read() for _ in range(st["case"]["n_it"])] + [g.step_read_flush()]
    got = np.array([p for p in got if p is not None])
    return dict(i=got[:, 0], var=got[:, 1])


def _run_parts(st):
    g, buf, case = st["g"], st["buf"], st["case"]
    for p in range(case["parts"]):
        g.iterate_part(p, case["parts"])
    g.export_partials(buf.data_ptr())
    g.import_partials(buf.data_ptr())
    g.estimate()
    g.adapt()
    n, m = g.n_hc, case["dim"] * case["n_g"]
    return dict(s1=buf[:n], s2=buf[n:2 * n], hsum=buf[2 * n:2 * n + m], hcnt=buf[2 * n + m:])


def _run_batch(st):
    case = st["case"]
    b = vegasp.Batch(st["members"], precision=PREC[case["precision"]])
    b.run(case["n_it"])
    rs = b.results(discard=case["n_it"] // 3)
    b.close()
    return {k: np.array([r[k] for r in rs], np.float32) for k in ("mean", "last_i")}


def _run_serve(st):
    case, s = st["case"], st["server"]
    for tag, prob in enumerate(st["requests"]):
        # (a target nothing reaches: every request runs its n_it iterations)
        s.submit(prob, rtol=1e-12, discard=case["n_it"] // 2, max_it=case["n_it"],
                 precision=PREC[case["precision"]], tag=tag)
    while s.step() > 0:
        pass
    got = sorted(s.poll(len(st["requests"])), key=lambda r: r["tag"])
    # (a posterior's integral is its evidence, quoted as its logarithm)
    return dict(log_evidence=np.log([r["mean"] for r in got]).astype(np.float32),
                n_iter=np.array([r["n_iter"] for r in got], np.int64))


def _run_alloc(st):
    case = st["case"]
    p = ctypes.c_void_p
    vegasp.check(vegasp.lib().vp_alloc_static(
        p(st["d"].data_ptr()), case["n_hc"], case["n_ev"], int(case["plus2"]),
        p(st["n"].data_ptr()), p(st["off"].data_ptr()), vegasp.current_stream()))
    return dict(n_h=st["n"], offsets=st["off"])


RUN = {"job": _run_job, "production": _run_production, "parts": _run_parts, "batch": _run_batch,
       "serve": _run_serve, "alloc": _run_alloc}


def run(state):
    return RUN[state["case"]["call"]](state)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _strata(dim, n_ev, mixed=False):
    """§3 Eq. (Nst_vegasp): the largest n with 4 n^dim <= n_ev on every axis;
    mixed (§3.2): n + 1 on as many leading axes as 4 samples a hypercube allow."""
    n = 1
    while 4 * (n + 1) ** dim <= n_ev:
        n += 1
    s = [n] * dim
    if mixed:
        d = 0
        while d < dim and 4 * (n + 1) ** (d + 1) * n ** (dim - d - 1) <= n_ev:
            d += 1
        s = [n + 1] * d + [n] * (dim - d)
    return s


def _iteration_work(dim, n_ev, n_g, family, peaks=1, points=50, outputs=1, mixed=False):
    """Algorithmic operations and bytes of one iteration: per sample the map (4
    an axis), the integrand, the moments (10) and the histogram sums (one an
    axis); per hypercube the allocation read and written once; the grid read
    and written once."""
    if family == "posterior":
        par = 2
        f = points * (2 * par + 10) + 2 * par + 1
    else:
        f = peaks * (3 * dim + {"gauss": 2, "ball": 1, "exp": 3}[family])
    if outputs > 1:
        f += 3 * outputs + outputs * (outputs + 1)
    n_hc = math.prod(_strata(dim, n_ev, mixed))
    return n_ev * (4 * dim + f + 10 + dim), 8 * n_hc + 16 * dim * n_g


def work(case):
    call = case["call"]
    if call == "alloc":
        return dict(bytes=20.0 * case["n_hc"], flops=2.0 * case["n_hc"])
    parts = []
    if call == "batch":
        # (the members are drawn with the inputs: the mean over their ranges)
        lo, hi = case["n_ev_lo"], case["n_ev_hi"]
        n_ev = int((hi - lo) / math.log(hi / lo)) if hi > lo else lo
        dim = (case["dim_lo"] + case["dim_hi"]) // 2
        parts.append((case["members"] * case["n_it"],
                      _iteration_work(dim, n_ev, case["n_g"], "gauss", peaks=2.5)))
    elif call == "serve":
        k = case["share_d21"]
        for share, dim, n_ev in ((1 - k, 3, case["n_ev_d3"]), (k, 21, case["n_ev_d21"])):
            parts.append((case["requests"] * case["n_it"] * share,
                          _iteration_work(dim, n_ev, case["n_g"], "posterior")))
    else:
        parts.append((case.get("n_it", 1), _iteration_work(
            case["dim"], case["n_ev"], case["n_g"], case["family"], case.get("peaks", 1),
            case.get("points", 50), case.get("outputs", 1), case.get("mixed", False))))
    return dict(flops=float(sum(n * w[0] for n, w in parts)),
                bytes=float(sum(n * w[1] for n, w in parts)))


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the paper's formulas in plain torch
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words (a product's high
    half survives the wrap: arithmetic shift, then mask)."""
    k0, k1 = key
    for _ in range(10):
        p, q = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((q >> 32) & M32) ^ c[1] ^ k0, q & M32, ((p >> 32) & M32) ^ c[3] ^ k1, p & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _integrand(prob, x):
    """f at the points x[axis] (tensors), 64 bits."""
    prm = prob.prm
    if prob.kind == inputs.POSTERIOR:
        n, P, G = int(prm[0]), int(prm[1]), int(prm[2])
        sy, pw, ref = prm[3:6]
        y, A = prm[6:6 + n], prm[6 + n:].reshape(n, P)
        s2pi = math.sqrt(2.0 * math.pi)
        lg = torch.zeros_like(x[0])
        for i in range(n):
            w = x[P + i % G]
            r2 = (y[i] - sum(A[i, m] * x[m] for m in range(P))) ** 2
            lg += torch.log((1.0 - w) / (s2pi * sy) * torch.exp(-r2 / (2.0 * sy * sy)) +
                            w / (s2pi * 10.0 * sy) * torch.exp(-r2 / (200.0 * sy * sy)))
        for m in range(P):
            lg -= x[m] ** 2 / (2.0 * pw * pw)
        return torch.exp(lg - ref)
    f = torch.zeros_like(x[0])
    for row in prm[1:].reshape(int(prm[0]), 2 + prob.dim):
        r2 = sum((x[m] - row[2 + m]) ** 2 for m in range(prob.dim))
        if prob.kind == inputs.GAUSS:
            f += row[0] * torch.exp(-r2 / row[1] ** 2)
        elif prob.kind == inputs.BALL:
            f += row[0] * (r2 < row[1] ** 2)
        else:
            f += row[0] * torch.exp(-row[1] * torch.sqrt(r2))
    return f


class _Plain:
    """One vegas+ integral in 64 bits on the points the library documents: u
    from one 32-bit Philox word, (r + 1/2) 2^-32, or its top 23 bits on the
    FP32 path, ((r >> 9) + 1/2) 2^-23."""

    def __init__(self, prob, precision, edges=None, mono=None):
        self.p, self.fp32 = prob, precision == "fp32"
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        D, G = prob.dim, prob.n_g
        if edges is None:
            lo, hi = np.asarray(prob.lo, float)[:, None], np.asarray(prob.hi, float)[:, None]
            edges = lo + (hi - lo) * np.arange(G + 1)[None, :] / G
        self.edges = torch.from_numpy(np.ascontiguousarray(edges)).to(self.dev)
        self.s = _strata(D, prob.n_ev, prob.mixed)
        self.n_hc = math.prod(self.s)
        n0 = max(2, prob.n_ev // self.n_hc)
        self.n_h = torch.full((self.n_hc,), n0, dtype=torch.int64, device=self.dev)
        self.mono = None if not mono else [(-1, -1)] + list(mono)
        self.t, self.I, self.V, self.Im, self.Cm = 0, [], [], [], []

    def sample(self, hist):
        p, D, G, dev = self.p, self.p.dim, self.p.n_g, self.dev
        z = lambda *n: torch.zeros(*n, dtype=torch.float64, device=dev)  # noqa: E731
        self.s1, self.s2 = z(self.n_hc), z(self.n_hc)
        self.hs, self.hc = z(D, G), z(D, G)
        M = len(self.mono) if self.mono else 0
        self.x1, self.x2 = z(self.n_hc, M), z(self.n_hc, M, M)
        off = torch.zeros(self.n_hc + 1, dtype=torch.int64, device=dev)
        off[1:] = torch.cumsum(self.n_h, 0)
        total, calls = int(off[-1]), (D + 3) // 4
        key = (p.seed & M32, (p.seed >> 32) & M32)
        step = 4_000_000 if dev == "cuda" else 400_000
        for a in range(0, total, step):
            k = torch.arange(a, min(a + step, total), device=dev)
            h = torch.searchsorted(off, k, right=True) - 1
            j, rest = k - off[h], h.clone()
            jac = torch.ones(k.numel(), dtype=torch.float64, device=dev)
            x, idx = [], []
            for q in range(calls):
                w = _philox([(j * calls + q) & M32, h, torch.full_like(h, self.t),
                             torch.full_like(h, p.integral_id)], key)
                for mu in range(4 * q, min(4 * q + 4, D)):
                    r = w[mu - 4 * q]
                    u = ((r >> 9).double() + 0.5) * 2.0 ** -23 if self.fp32 else \
                        (r.double() + 0.5) * 2.0 ** -32
                    y = ((rest % self.s[mu]).double() + u) / self.s[mu]
                    rest = rest // self.s[mu]
                    i = torch.clamp((y * G).long(), max=G - 1)
                    e0 = self.edges[mu][i]
                    dx = self.edges[mu][i + 1] - e0
                    x.append(e0 + dx * (y * G - i))
                    jac *= G * dx
                    idx.append(i)
            v = jac * _integrand(p, x)
            self.s1.index_add_(0, h, v)
            self.s2.index_add_(0, h, v * v)
            if hist:
                d = v * v / self.n_h[h] if p.d_weighted else v * v
                for mu in range(D):
                    self.hs[mu].index_add_(0, idx[mu], d)
                    self.hc[mu].index_add_(0, idx[mu], torch.ones_like(d))
            if M:
                one = torch.ones_like(v)
                vk = torch.stack([v * (one if b < 0 else x[b]) * (one if c < 0 else x[c])
                                  for b, c in self.mono], 1)
                self.x1.index_add_(0, h, vk)
                self.x2.index_add_(0, h, vk[:, :, None] * vk[:, None, :])

    def estimate(self):
        n, om = self.n_h.double(), 1.0 / self.n_hc
        m1 = self.s1 / n
        var = torch.clamp(self.s2 / n - m1 * m1, min=0.0)
        self.I.append(float(om * m1.sum()))
        self.V.append(float(om * om * (var / (n - 1)).sum()))
        if self.mono:
            mk = self.x1 / n[:, None]
            c = self.x2 / n[:, None, None] - mk[:, :, None] * mk[:, None, :]
            diag = torch.eye(len(self.mono), dtype=torch.bool, device=self.dev)
            c = torch.where(diag & (c < 0), torch.zeros_like(c), c)
            self.Im.append((om * mk.sum(0)).cpu().numpy())
            self.Cm.append((om * om * (c / (n - 1)[:, None, None]).sum(0)).cpu().numpy())
        self.d = (om * torch.sqrt(var)) ** self.p.beta
        self.t += 1

    def allocate(self):
        q = self.p.n_ev * self.d / self.d.sum()
        self.n_h = torch.clamp(torch.floor(q * (1.0 + 2.0 ** -50)).long(), min=2)

    def refine(self):
        p, G = self.p, self.p.n_g
        d = self.hs if p.d_weighted else torch.where(self.hc > 0, self.hs / self.hc,
                                                     torch.zeros_like(self.hs))
        tot = d.sum(1, keepdim=True)
        s = torch.empty_like(d)
        s[:, 0] = (7.0 * d[:, 0] + d[:, 1]) / 8.0
        s[:, 1:-1] = (d[:, :-2] + 6.0 * d[:, 1:-1] + d[:, 2:]) / 8.0
        s[:, -1] = (d[:, -2] + 7.0 * d[:, -1]) / 8.0
        s = torch.clamp(s / tot, min=2.2250738585072014e-308)
        c = torch.where(s < 1.0, ((1.0 - s) / -torch.log(s)) ** p.alpha, torch.ones_like(s))
        for mu in range(p.dim):
            if not float(tot[mu]) > 0.0:
                continue
            cum = torch.cumsum(c[mu], 0)
            want = cum[-1] * torch.arange(1, G, dtype=torch.float64, device=self.dev) / G
            k = torch.clamp(torch.searchsorted(cum, want), max=G - 1)
            e = self.edges[mu].clone()
            self.edges[mu][1:G] = e[k + 1] - (cum[k] - want) / c[mu][k] * (e[k + 1] - e[k])

    def iterate(self, adapt):
        self.sample(hist=adapt)
        self.estimate()
        self.allocate()
        if adapt:
            self.refine()


def exact(case, seed):
    call = case["call"]
    if call == "alloc":
        d = _alloc_d(case, seed)
        q = case["n_ev"] * d / math.fsum(d)
        n = np.floor(q * (1.0 + 2.0 ** -50)).astype(np.int64)
        n = n + 2 if case["plus2"] else np.maximum(n, 2)
        return dict(n_h=n.astype(np.int32), offsets=np.concatenate([[0], np.cumsum(n)]))
    if call in ("batch", "serve"):  # (hundreds of integrals: minutes this way)
        return None
    prob = _problem(case, seed)
    if call == "job":
        mono = _monomials(case["outputs"]) if case.get("outputs", 1) > 1 else None
        v = _Plain(prob, case["precision"], mono=mono)
        for _ in range(case["n_it"]):
            v.iterate(adapt=True)
        out = dict(i=np.array(v.I), sdev=np.sqrt(v.V), edges=v.edges.cpu().numpy())
        if mono:
            out["i_multi"], out["cov_multi"] = np.array(v.Im), np.array(v.Cm)
        if case["precision"] == "fp64":
            i, w = np.array(v.I[2:]), 1.0 / np.array(v.V[2:])
            out["mean"] = float((w * i).sum() / w.sum())
            out["n_h"] = v.n_h.cpu().numpy()
        return out
    v = _Plain(prob, case["precision"], edges=_trained_grid(prob))
    if call == "parts":
        v.sample(hist=True)
        return dict(s1=v.s1, s2=v.s2, hsum=v.hs, hcnt=v.hc)
    for _ in range(case["n_it"]):
        v.iterate(adapt=False)
    return dict(i=np.array(v.I), var=np.array(v.V))
