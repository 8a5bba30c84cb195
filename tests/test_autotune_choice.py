"""The autotuner's choice between the sorts: a cached one is a preference where
the call sorts (2, 3), anything else is left alone (host logic, no GPU); and
on a GPU a tuned setting passed back as it is does not make a call sort that
is faster without."""
import pytest

from paper_2203_02527_gb300 import autotune, ph0


@pytest.mark.parametrize("stored,applied", [(0, 2), (1, 3), (-1, -1), (2, 2), (3, 3), (None, -1)])
def test_cached_choice(monkeypatch, stored, applied):
    t = {"dist_tile": 64} if stored is None else {"dist_tile": 64, "packed_sort": stored}
    monkeypatch.setattr(autotune, "cached", lambda d, n: dict(t))
    got = ph0._tuning(5000, 3, None)
    assert got.packed_sort == applied and got.dist_tile == 64


@pytest.mark.gpu
@pytest.mark.parametrize("d,n", [(16, 8192), (3, 6000), (8, 2000)])
def test_tuned_setting_passed_back(tmp_path, monkeypatch, d, n):
    import torch

    from paper_2203_02527_gb300 import inputs
    monkeypatch.setenv("PH0_TUNING_CACHE", str(tmp_path / "tuning.json"))
    monkeypatch.setattr(autotune, "_cache", None)
    t = autotune.tune(d, n=n, repeats=2)
    assert "packed_sort" not in t
    x = torch.from_numpy(inputs.uniform(n, d, seed=98)).cuda()
    got, want = ph0.barcodes(x, tuning=t), ph0.barcodes(x, tuning={"packed_sort": 0})
    assert got.stats["sort_form"] == 3 and torch.equal(got.raw, want.raw)
