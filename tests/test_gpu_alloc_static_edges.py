"""vp_alloc_static at the edges of its blocks, on buffers that start on a 16-byte
boundary (vector loads and stores) or one element past it (scalar ones), and
with N_ev near 2^32 (a block's samples pass 2^32): bit for bit the oracle's
reallocation (§3 Eq. nh), the bytes around the buffers untouched."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_hc", [1, 3, 1023, 1025, 262_145, (1 << 22) - 3])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n_ev,plus2", [(10_000_019, False), (4_294_967_293, True)])
def test_alloc_static_edges(n_hc, shift, n_ev, plus2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2009_05112_gb300 import build
    build.build()
    from paper_2009_05112_gb300 import vegasp as V
    rng = np.random.default_rng(n_hc + shift)
    d = rng.exponential(size=n_hc) * 10.0 ** rng.uniform(-8, 8, size=n_hc)
    d[rng.uniform(size=n_hc) < 0.2] = 0.0
    d[0] = max(d[0], 10.0 * d.sum() + 1.0)  # most of the samples in one hypercube
    pad = 4
    d_dev = torch.zeros(n_hc + 2 * pad, dtype=torch.float64, device="cuda")
    n_dev = torch.full((n_hc + 2 * pad,), -7, dtype=torch.int32, device="cuda")
    o_dev = torch.full((n_hc + 1 + 2 * pad,), -7, dtype=torch.int64, device="cuda")
    at = pad + shift
    d_dev[at:at + n_hc] = torch.from_numpy(d).cuda()
    p = ctypes.c_void_p
    for _ in range(2):
        V.check(V.lib().vp_alloc_static(p(d_dev[at:].data_ptr()), n_hc, n_ev, int(plus2),
                                        p(n_dev[at:].data_ptr()), p(o_dev[at:].data_ptr()),
                                        V.current_stream()))
    n_ref, off_ref = oracle.allocate(n_ev, d, plus2=plus2)
    n_got, o_got = n_dev.cpu().numpy(), o_dev.cpu().numpy()
    assert np.array_equal(n_got[at:at + n_hc].view(np.uint32), n_ref)
    assert np.array_equal(o_got[at:at + n_hc + 1].view(np.uint64), off_ref)
    assert np.all(n_got[:at] == -7) and np.all(n_got[at + n_hc:] == -7)
    assert np.all(o_got[:at] == -7) and np.all(o_got[at + n_hc + 1:] == -7)
