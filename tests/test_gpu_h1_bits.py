"""First homology's columns as bit sets: more columns than are reduced at a
time (several batches), against the oracle's literal reduction bit for bit,
and the structure of the result on both sides of the largest size of that form."""
import numpy as np
import pytest

from paper_2203_02527_gb300 import inputs
from tests.test_gpu_h1 import _check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(220, 8), (257, 16)])
def test_batches_of_columns(n, d):
    assert _check(inputs.uniform(n, d, seed=60 + n))["reduced"] > 128


@pytest.mark.parametrize("n", [1024, 1025])
def test_largest_bit_sets(n):
    from paper_2203_02527_gb300 import ph0
    x = torch.from_numpy(inputs.uniform(n, 2, seed=61)).cuda()
    bars, st = ph0.h1(x)
    m = n * (n - 1) // 2
    assert st["n_bars"] == len(bars) == m - (n - 1) and st["n_triangles"] == n * (n - 1) * (n - 2) // 6
    h0 = ph0.barcodes(x).numpy()
    births = set(zip(bars["eu"].tolist(), bars["ev"].tolist()))
    killing = set(zip(h0["u"].tolist(), h0["v"].tolist()))
    assert len(births) == len(bars) and births.isdisjoint(killing) and len(births) + len(killing) == m
    assert (bars["death_order"] > bars["birth_order"])[bars["death_sq"] > bars["birth_sq"]].all()
    assert (np.diff(bars["death_rank"]) > 0).all()
