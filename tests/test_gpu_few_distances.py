"""Clouds whose points or distances repeat in their thousands, above the sizes
of the distance matrix: the form without a sort gives the sorted form's bars
bit for bit (integers, so there is no tolerance), and none of its steps takes
as long as a good part of that form's whole path, measured side by side on the
same GPU (a step that waits for millions of atomics on one word takes longer
than all of it)."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 20000


def copies(n, r):
    """n points, r shuffled copies of each of n / r."""
    rng = np.random.default_rng(71)
    x = np.repeat(rng.random((n // r, 3)).astype(np.float32), r, axis=0)
    return x[rng.permutation(len(x))]


def halves(n, shuffled):
    x = np.zeros((n, 2), np.float32)
    x[np.random.default_rng(72).permutation(n)[:n // 2] if shuffled else np.arange(n // 2)] = 1.0
    return x


def hot(n, k):
    """k copies of one point among uniform ones."""
    rng = np.random.default_rng(73)
    x = rng.random((n, 3)).astype(np.float32)
    x[rng.permutation(n)[:k]] = 0.5
    return x


def line_and_plane(n, places):
    """Half of n points at whole places on a line, half in the plane, in random order."""
    rng = np.random.default_rng(75)
    x = rng.random((n, 2)).astype(np.float32) * places
    at = rng.permutation(n)[:n // 2]
    x[at, 0], x[at, 1] = rng.integers(0, places, len(at)), 0.0
    return x


def signed(x):
    """Some of the zeros negative."""
    return np.where((x == 0) & (np.random.default_rng(76).random(x.shape) < 0.5), np.float32(-0.0), x)


CLOUDS = {
    "two_points": lambda: halves(N, True),
    "two_points_in_order": lambda: halves(N, False),
    "cube_corners": lambda: np.random.default_rng(74).integers(0, 2, (N, 3)).astype(np.float32),
    "copies_256": lambda: copies(N, 256),
    "copies_64": lambda: copies(N, 64),
    "copies_16": lambda: copies(N, 16),
    "a_fifth_equal": lambda: hot(N, N // 5),
    "half_on_a_line_50000": lambda: line_and_plane(50000, 300),
    "a_fifth_equal_50000": lambda: hot(50000, 10000),
    "uniform_50000": lambda: hot(50000, 1),
    "one_point": lambda: np.full((N, 2), 0.25, np.float32),
    "two_points_5000": lambda: halves(5000, True),
    "signed_zeros_5000": lambda: signed(halves(5000, True)),
    "copies_4_5000": lambda: copies(5000, 4),
    "copies_64_5000": lambda: copies(5000, 64),
    "one_point_5000": lambda: np.full((5000, 2), 0.25, np.float32),
}


@functools.lru_cache(maxsize=None)
def measured(name):
    """Both forms' bars and least stage times of four runs."""
    from paper_2203_02527_gb300 import ph0
    x = torch.from_numpy(np.ascontiguousarray(CLOUDS[name]())).cuda()
    out = []
    for tuning in (None, {"packed_sort": 0}):
        runs = [ph0.barcodes_profiled(x, tuning=tuning) for _ in range(4)]
        times = {k: min(p[k] for _, p in runs[1:]) for k in ("total_ms", "reduce_ms", "dedupe_ms", "sort_ms")}
        out.append((ph0.barcodes(x, tuning=tuning), times))
    torch.cuda.empty_cache()
    return x, out


@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_bars(name):
    x, ((got, _), (want, _)) = measured(name)
    assert got.stats["sort_form"] == 3 and want.stats["sort_form"] in (0, 2)
    assert torch.equal(got.raw, want.raw) and got.inf == want.inf
    assert got.stats["n_distinct"] == want.stats["n_distinct"]


@pytest.mark.parametrize("name", sorted(k for k in CLOUDS if "000" not in k))
def test_early_path(name):
    from paper_2203_02527_gb300 import ph0
    x, ((want, _), _) = measured(name)
    got = ph0.barcodes_early(x)
    assert got.stats["sort_form"] == 3
    assert torch.equal(got.raw, want.raw) and got.inf == want.inf
    assert got.stats["n_distinct"] == int(want.a[-1])


@pytest.mark.parametrize("name", ["two_points", "two_points_in_order", "cube_corners", "copies_256", "two_points_5000"])
def test_tree_among_equal_distances(name):
    """The tree and its pivots: less than half the sorted form's whole path."""
    _, ((_, form), (_, whole)) = measured(name)
    assert form["reduce_ms"] < 0.5 * whole["total_ms"], (form, whole)


@pytest.mark.parametrize("name", ["two_points", "two_points_in_order", "cube_corners", "copies_256", "two_points_5000"])
def test_counts_among_equal_distances(name):
    """The counts and the repeated distances: less than half the sorted form's whole path."""
    _, ((_, form), (_, whole)) = measured(name)
    assert form["dedupe_ms"] < 0.5 * whole["total_ms"], (form, whole)


def test_distances_repeated_among_distinct_ones():
    """16,000 distances that come ten thousand times each, too few of one in a
    tile of 8,192 edges to be taken out there, in buckets of ten thousand
    others: the counts and the repeated distances take less than 2.5 times as
    long as without any repeated (a bucket is not read once per 5,000 keys)."""
    _, ((_, form), _) = measured("a_fifth_equal_50000")
    _, ((_, plain), _) = measured("uniform_50000")
    assert form["dedupe_ms"] < 2.5 * plain["dedupe_ms"], (form, plain)


@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_whole_path(name):
    """The whole path: no longer than the sorted form's, but for the runs'
    differences (a quarter: the least of three of each, side by side)."""
    _, ((_, form), (_, whole)) = measured(name)
    assert form["total_ms"] < 1.25 * whole["total_ms"], (form, whole)
