"""vp_alloc_static where the product N_ev d_h or N_ev sum d leaves the doubles,
and on d_h outside the documented range: the quotient as written, N_ev d_h then
divided by the sum, floored, as an unsigned 32-bit number.  Every d_h is a whole
multiple of one power of two, so that the sum is exact in any order."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def expected(d, n_ev, plus2):
    s = float(d.sum())
    with np.errstate(over="ignore", invalid="ignore"):
        q = np.float64(n_ev) * d / s if s > 0 else np.full(d.size, np.float64(n_ev) / d.size)
        fl = np.floor(q)
        fl = np.where((fl + 1.0) - q <= q * 2.0 ** -50, fl + 1.0, fl)
    u = np.clip(fl, 0.0, 4294967295.0).astype(np.uint64)
    n = (u + 2) % (1 << 32) if plus2 else np.where(fl > 2.0, u, 2)
    return n.astype(np.uint32)


def whole(rng, n, top, unit):
    return np.ldexp(rng.integers(0, top, n).astype(float), unit)


def cases():
    rng = np.random.default_rng(3)
    a = whole(rng, 20_000, 1 << 20, 984)        # N_ev sum d overflows, no N_ev d_h does
    a[rng.random(a.size) < 0.98] = 0.0
    yield "overflowing sum", a, 20_011
    b = whole(rng, 3000, 1 << 20, 985)          # ... and one N_ev d_h does
    b[7] = np.ldexp(1.0, 1020)
    yield "overflowing product", b, 100_003
    c = whole(rng, 5000, 1 << 20, 0)
    c[::7] *= -1.0                              # (a zero among them becomes -0)
    yield "negative", c, 1_000_003
    d = whole(rng, 5000, 1 << 20, 0) * -1.0
    d[11] = 2.0 - (d.sum() - d[11])             # quotients far beyond 32 bits, sum d = 2
    yield "larger than the sum", d, 4_000_000_007
    yield "negative sum", whole(rng, 3000, 1 << 20, 0) * -1.0, 100_003
    yield "negative sum, overflowing", whole(rng, 20_000, 1 << 20, 980) * -1.0, 100_003


@pytest.mark.parametrize("name,d,n_ev", list(cases()), ids=[c[0] for c in cases()])
@pytest.mark.parametrize("plus2", [False, True])
def test_quotient_as_written(name, d, n_ev, plus2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05112_gb300 import build
    build.build()
    from paper_2009_05112_gb300 import vegasp as V
    p = ctypes.c_void_p
    t = torch.from_numpy(d).cuda()
    n_dev = torch.zeros(d.size, dtype=torch.int32, device="cuda")
    o_dev = torch.zeros(d.size + 1, dtype=torch.int64, device="cuda")
    V.check(V.lib().vp_alloc_static(p(t.data_ptr()), d.size, n_ev, int(plus2),
                                    p(n_dev.data_ptr()), p(o_dev.data_ptr()), V.current_stream()))
    n = expected(d, n_ev, plus2)
    assert np.array_equal(n_dev.cpu().numpy().view(np.uint32), n)
    assert np.array_equal(o_dev.cpu().numpy().view(np.uint64),
                          np.concatenate([[0], np.cumsum(n.astype(np.uint64))]).astype(np.uint64))
