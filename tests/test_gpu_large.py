"""The whole path without a sort above 2896 points against the oracle, every
field of every bar bit for bit (positions, indices and keys are integers, so
there is no tolerance): at the edges of its range, of the partitions that are
looked at without buckets (12.6M edges), of the counts kept in shared memory
(8192 killing edges); on ties, duplicate points, wide exponents, crowded
distances, and clouds whose tree the list of short edges does not reach."""
import numpy as np
import pytest

from paper_2203_02527_gb300 import inputs
from tests.test_gpu_direct import _chain, check

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(2897, 1), (2898, 2), (3000, 3), (4096, 3), (5016, 2), (5017, 2), (5018, 3), (4345, 5), (5794, 5),
                                 (8192, 2), (8193, 3), (8200, 8)])
def test_sizes(n, d):
    check(inputs.uniform(n, d, seed=3400 + n))


@pytest.mark.parametrize("name", ["lattice", "lattice3", "lattice3_20", "bytes", "one_point", "integers", "duplicates", "exponents",
                                  "signed_zeros", "chain", "crowded", "outliers", "mixture"])
def test_clouds(name):
    rng = np.random.default_rng(3500)
    crowded = rng.random((3200, 3)) * 1e-12
    crowded[1600:, 1] = 1.0
    x = {"lattice": lambda: inputs.lattice(75, 2), "lattice3": lambda: inputs.lattice(15, 3),
         "lattice3_20": lambda: inputs.lattice(20, 3),
         "bytes": lambda: rng.integers(0, 256, (6000, 3)).astype(np.float32),
         "one_point": lambda: np.full((3000, 2), 0.5, np.float32),
         "integers": lambda: rng.integers(0, 3000, (5200, 1)).astype(np.float32),
         "duplicates": lambda: inputs.with_duplicates(3100, 3, 700, seed=3501),
         "exponents": lambda: inputs.exponent_gaps(3000, 3, seed=3502),
         "signed_zeros": lambda: inputs.negative_zero_mix(3000, 3, seed=3503),
         "chain": lambda: _chain(3000),
         "crowded": lambda: crowded.astype(np.float32),
         "outliers": lambda: inputs.circles_with_outliers(1500, 4, 16, 4, seed=3504),
         "mixture": lambda: inputs.gaussian_mixture(6000, 3, k=8, sigma=0.05, center_range=10.0, seed=3505)}[name]()
    check(x)


@pytest.mark.parametrize("name", ["uniform3", "line", "lattice", "mixture", "circles", "one_point"])
def test_early_path_keeps_only_the_prefix(name):
    """From 2^27 edges on the early path counts repeated distances only up to
    the last killing edge: the whole path's bars, the prefix's length and its
    number of distinct distances (the last bar's a, or more with ties)."""
    import torch

    from paper_2203_02527_gb300 import ph0
    x = {"uniform3": lambda: inputs.uniform(16400, 3, seed=3601),
         "line": lambda: inputs.uniform(16500, 1, seed=3602),
         "lattice": lambda: inputs.lattice(26, 3),
         "mixture": lambda: inputs.gaussian_mixture(16411, 5, k=8, sigma=0.05, center_range=10.0, seed=3603),
         "circles": lambda: inputs.circles_with_outliers(4100, 4, 16, 3, seed=3604),
         "one_point": lambda: np.full((16390, 2), 0.5, np.float32)}[name]()
    pts = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    whole, early = ph0.barcodes(pts), ph0.barcodes_early(pts)
    assert torch.equal(early.raw, whole.raw) and early.inf == whole.inf
    bars, m = whole.numpy(), len(x) * (len(x) - 1) // 2
    assert early.stats["sort_form"] == 3
    assert int(bars["order"][-1]) < early.stats["sorted_edges"] <= m
    assert early.stats["n_distinct"] == int(bars["a"][-1]) <= whole.stats["n_distinct"]
    torch.cuda.empty_cache()
