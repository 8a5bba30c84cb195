"""Buckets of repeated distances whose distinct keys do not fit their table
are taken in halves by bits of the hash (csrc/k_direct.cu, csrc/k_large.cu).
With the library's tables only keys that a hash crowds on purpose would show
it, so this builds both units with so few probes that nearly every bucket is
halved several times, and compares every field of every bar with the oracle
(integers and keys, so there is no tolerance)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal
from tests.variants import build_variant

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def few_probes(tmp_path_factory):
    return build_variant(tmp_path_factory.mktemp("few_probes"), ("k_direct", "k_large"),
                         ["-DPH0_DIR_PROBES=3", "-DPH0_LG_PROBES=4"])


def _cases():
    rng = np.random.default_rng(81)
    copies = np.repeat(rng.random((2500, 3)), 2, axis=0)[rng.permutation(5000)]
    return {
        "uniform_1500": inputs.uniform(1500, 3, seed=82),                          # buckets of 4,096 keys
        "uniform_2896": inputs.uniform(2896, 2, seed=83),                          # of 8,192
        "integers_2500": rng.integers(0, 100, (2500, 2)),                          # buckets beyond their room
        "lattice_60": inputs.lattice(60, 2),                                       # few distances, large buckets
        "bytes_6000": rng.integers(0, 256, (6000, 3)),
        "copies_5000": copies,
    }


@pytest.mark.parametrize("name", sorted(_cases()))
def test_halved_buckets(few_probes, name):
    from paper_2203_02527_gb300 import _lib, ph0
    x = np.ascontiguousarray(_cases()[name], np.float32)
    n, d = x.shape
    pts, ws = torch.from_numpy(x).cuda(), ph0.Workspace(n, d)
    raw = torch.empty((n - 1, _lib.BAR_BYTES), dtype=torch.uint8, device="cuda")
    st = _lib.Stats()
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert few_probes.ph0_barcodes_tuned(pts.data_ptr(), n, d, d, raw.data_ptr(), None, ws.ptr, ws.nbytes, stream,
                                         None) == 0
    assert few_probes.ph0_finish(ws.ptr, stream, ctypes.byref(st)) == 0
    want, _, distinct = oracle.barcodes(x)
    assert_bars_equal(raw.cpu().numpy().reshape(-1).view(_lib.BAR_DTYPE), want)
    assert st.sort_form == 3 and st.n_distinct == distinct
