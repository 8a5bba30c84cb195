"""First homology when the room for reduced columns runs out, on a build that
has little of it: the call reports PH0_ETOOBIG without delay (a column that
found no room claims nothing, so no later one adds an empty column over and
over), and the library's own build then computes the same cloud."""
import ctypes
import time

import pytest

from paper_2203_02527_gb300 import inputs
from tests.test_gpu_h1 import _check
from tests.variants import build_variant

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small_pool(tmp_path_factory):
    return build_variant(tmp_path_factory.mktemp("small_pool"), ("k_h1", "ph0_capi"), ["-DPH0_H1_POOL=200"])


@pytest.mark.parametrize("n,d", [(220, 8), (150, 3)])
def test_full_pool(small_pool, n, d):
    from paper_2203_02527_gb300 import _lib
    x = inputs.uniform(n, d, seed=60 + n)
    pts = torch.from_numpy(x).cuda()
    nbytes = int(small_pool.ph0_h1_workspace_bytes(n, d))
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    m = n * (n - 1) // 2
    bars = torch.empty((m - (n - 1), _lib.H1_BAR_BYTES), dtype=torch.uint8, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    st = _lib.H1Stats()
    for _ in range(2):
        t0 = time.perf_counter()
        rc = small_pool.ph0_h1(pts.data_ptr(), n, d, d, bars.data_ptr(), ws.data_ptr(), nbytes, stream,
                               ctypes.byref(st))
        assert rc == 3 and time.perf_counter() - t0 < 0.5  # PH0_ETOOBIG
    _check(x)
