"""vp_alloc_static after a call of it that failed between its launches: the next
call answers as if that one had not been.  The launch that fails is a fake of
cudaLaunchKernelEx compiled over the library's own source; the launches before
it run as they are."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WRAP = r"""
#include <cuda_runtime.h>
static int g_left = -1;  // launches until the one that fails (-1: none does)
template <class... K, class... A>
static cudaError_t fake_launch(const cudaLaunchConfig_t *c, void (*k)(K...), A... a) {
    if (g_left >= 0 && g_left-- == 0) return cudaErrorLaunchOutOfResources;
    return cudaLaunchKernelEx(c, k, a...);
}
#define cudaLaunchKernelEx fake_launch
#include "noalloc.cu"
namespace vp {
const char *set_error_message(vp_status, const char *m) { return m; }
}
extern "C" void fail_after(int n) { g_left = n; }
"""


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05112_gb300 import build
    d = tmp_path_factory.mktemp("faked")
    src, so = str(d / "faked.cu"), str(d / "libfaked.so")
    with open(src, "w") as f:
        f.write(WRAP)
    flags = [x for x in build.FLAGS if x != "-lineinfo"]
    subprocess.check_call([build._nvcc()] + build.ARCH + flags + ["-shared", "-o", so, src])
    return ctypes.CDLL(os.path.abspath(so))


@pytest.mark.parametrize("failing", [0, 1, 2])
@pytest.mark.parametrize("n_hc", [700, 40_000])
def test_next_call_recovers(faked, failing, n_hc):
    import oracle
    rng = np.random.default_rng(n_hc + failing)
    p = ctypes.c_void_p
    n_dev = torch.zeros(n_hc, dtype=torch.int32, device="cuda")
    o_dev = torch.zeros(n_hc + 1, dtype=torch.int64, device="cuda")

    def call(d, n_ev):
        t = torch.from_numpy(d).cuda()
        torch.cuda.synchronize()
        rc = faked.vp_alloc_static(p(t.data_ptr()), ctypes.c_int64(n_hc), ctypes.c_int64(n_ev), 0,
                                   p(n_dev.data_ptr()), p(o_dev.data_ptr()), p(0))
        torch.cuda.synchronize()
        return rc

    for n_ev in (1_000_003, 3_000_017):
        faked.fail_after(failing)
        assert call(rng.exponential(size=n_hc), 500_009) != 0
        faked.fail_after(-1)
        d = rng.exponential(size=n_hc) * 10.0 ** rng.uniform(-4, 4, size=n_hc)
        assert call(d, n_ev) == 0
        n_ref, off_ref = oracle.allocate(n_ev, d, plus2=False)
        assert np.array_equal(n_dev.cpu().numpy().view(np.uint32), n_ref)
        assert np.array_equal(o_dev.cpu().numpy().view(np.uint64), off_ref)
