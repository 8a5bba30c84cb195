"""The whole path without a sort (clouds of up to 2896 points) against the
oracle, every field of every bar bit for bit (positions, indices and keys are
integers, so there is no tolerance), at the edges of its tiles (32, 64 and 128
points a side), of its clusters (8 and 16 CTAs) and of its range; on ties,
duplicate points, crowded distances and chains of waiting columns; and the
sorted forms on the same clouds."""
import numpy as np
import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(x, tuning=None, form=3):
    from paper_2203_02527_gb300 import ph0
    want, inf_v, nd = oracle.barcodes(x)
    got = ph0.barcodes(torch.from_numpy(np.ascontiguousarray(x)).cuda(), tuning=tuning)
    assert_bars_equal(got.numpy(), want)
    assert got.inf == (inf_v, 0.0, float("inf"))
    assert got.stats["n_distinct"] == nd and got.stats["n_bars"] == len(x) - 1
    assert got.stats["sort_form"] == form
    return got


@pytest.mark.parametrize("n,d", [(2, 1), (3, 2), (7, 3), (8, 3), (9, 3), (31, 2), (32, 8), (33, 16), (63, 3), (65, 5),
                                 (128, 32), (512, 3), (513, 2), (1023, 3), (1024, 7), (1025, 3), (1999, 2), (2048, 8),
                                 (2049, 3), (2895, 1), (2896, 2), (100, 300), (40, 1024)])
def test_sizes(n, d):
    big = n == 40  # beyond the tile's room for coordinates: the short sort
    check(inputs.uniform(n, d, seed=3100 + n), form=0 if big else 3)


def _chain(n):
    # increasing gaps toward the first point: every column waits for the one before it
    gaps = np.arange(n, 1, -1, dtype=np.float64)
    return np.concatenate([[0.0], np.cumsum(gaps)])[:, None].astype(np.float32)


@pytest.mark.parametrize("name", ["lattice", "lattice3", "duplicates", "one_point", "exponents", "signed_zeros",
                                  "chain", "crowded", "circles", "simplex"])
def test_clouds(name):
    rng = np.random.default_rng(3200)
    crowded = rng.random((600, 3)) * 1e-12
    crowded[300:, 1] = 1.0
    x = {"lattice": lambda: inputs.lattice(33, 2), "lattice3": lambda: inputs.lattice(9, 3),
         "duplicates": lambda: inputs.with_duplicates(1100, 3, 90, seed=3201),
         "one_point": lambda: np.full((300, 2), 0.5, np.float32),
         "exponents": lambda: inputs.exponent_gaps(700, 4, seed=3202),
         "signed_zeros": lambda: inputs.negative_zero_mix(500, 3, seed=3203),
         "chain": lambda: _chain(900),
         "crowded": lambda: crowded.astype(np.float32),
         "circles": lambda: inputs.noisy_circles(300, 4, 16, seed=3204),
         "simplex": lambda: np.eye(130, dtype=np.float32)}[name]()
    check(x)


def test_rows_apart_and_the_sorted_forms():
    """Rows of 7 floats of which the first 3 count (a leading dimension above
    d), and the forms that sort, asked for on the same cloud."""
    from paper_2203_02527_gb300 import ph0
    x = inputs.uniform(777, 7, seed=3301)
    wide = torch.from_numpy(x).cuda()
    y = np.ascontiguousarray(x[:, :3])
    want = check(y).numpy()
    assert_bars_equal(ph0.barcodes(wide[:, :3]).numpy(), want)
    check(y, {"packed_sort": 0}, form=0)
    check(y, {"wide_ids": 1}, form=0)
    check(y, {"split_sort": 1}, form=0)
    bars, prof = ph0.barcodes_profiled(torch.from_numpy(y).cuda())
    assert_bars_equal(bars.numpy(), want)
    assert prof["total_ms"] > 0 and prof["dist_ms"] > 0 and prof["sort_ms"] == 0
