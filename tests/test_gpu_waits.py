"""Waits that run out, on each path that has one: the tree search of the early
path without a sort (tests/test_gpu_failures.py has the whole path's), the
reduction after a sort, and the early path's rounds.  The kernel gives up at
once with a limit of 0 and every later kernel of the call stays within its
buffers; the status is PH0_ETIMEOUT, and the same workspace then computes the
oracle's bars."""
import numpy as np
import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def timed_out(call):
    from paper_2203_02527_gb300._lib import Ph0Error
    with pytest.raises(Ph0Error) as e:
        call()
    assert e.value.code == 5  # PH0_ETIMEOUT


def test_early_path_without_a_sort():
    from paper_2203_02527_gb300 import ph0
    x = torch.from_numpy(inputs.uniform(16400, 2, seed=91)).cuda()
    ws = ph0.Workspace(16400, 2)
    want = ph0.barcodes(x)
    for _ in range(2):
        timed_out(lambda: ph0.barcodes_early(x, ws=ws, tuning={"reduce_spin_limit": 0}))
        got = ph0.barcodes_early(x, ws=ws)
        assert got.stats["sort_form"] == 3 and torch.equal(got.raw, want.raw) and got.inf == want.inf
    torch.cuda.empty_cache()


@pytest.mark.parametrize("sort", [{"packed_sort": 0}, {"packed_sort": 1}])
def test_reduction_after_a_sort(sort):
    from paper_2203_02527_gb300 import ph0
    x = inputs.uniform(4096, 4, seed=92)  # 64 reduction CTAs: some CTA always waits
    pts, ws = torch.from_numpy(x).cuda(), ph0.Workspace(4096, 4)
    timed_out(lambda: ph0.barcodes(pts, ws=ws, tuning={**sort, "reduce_spin_limit": 0}))
    got = ph0.barcodes(pts, ws=ws, tuning=sort)
    assert got.stats["sort_form"] == sort["packed_sort"]
    want, inf_v, nd = oracle.barcodes(x)
    assert_bars_equal(got.numpy(), want)
    assert got.stats["n_distinct"] == nd and got.inf[0] == inf_v
    assert np.array_equal(ph0.barcodes(pts, ws=ws).numpy()["order"], want["order"])
