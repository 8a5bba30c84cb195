"""The forms of the whole path that sort, asked for on clouds that run without
a sort by default, and the distance kernel's settings on every form that takes
them.  Every field of every bar against the oracle (integers and keys, so
there is no tolerance), and the form that ran: 0 the short sort, 2 the
complete sort after a fix-up met a group that it cannot order."""
import functools

import numpy as np
import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal
from tests.test_gpu_serving import _crowded_in

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run(x, tuning, form):
    from paper_2203_02527_gb300 import ph0
    want, inf_v, nd = oracle.barcodes(x)
    got = ph0.barcodes(torch.from_numpy(np.ascontiguousarray(x)).cuda(), tuning=tuning)
    assert got.stats["sort_form"] == form
    assert_bars_equal(got.numpy(), want)
    assert got.inf == (inf_v, 0.0, float("inf")) and got.stats["n_distinct"] == nd
    return got


def _simplex(n, spread, seed):
    rng = np.random.default_rng(seed)
    x = np.eye(n, dtype=np.float32)
    off = (rng.random((n, n)) * spread).astype(np.float32)
    np.fill_diagonal(off, 0)
    return (x + off).astype(np.float32)


def _two_clusters(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((2 * n, 3)) * 1e-12
    x[n:, 1] = 1.0
    return x.astype(np.float32)


def _two_pairs():
    x = inputs.uniform(3000, 3, seed=42)
    x[17], x[5] = x[2999], x[1234]
    return x


@pytest.mark.parametrize("name", ["groups_in_place", "one_long_group", "last_places", "many_tiles", "two_top_passes"])
def test_short_sort(name):
    """Groups of equal key >> 16 that the fix-up orders in place, one too long
    for it, distances that differ in the lowest byte only, a long group over
    1,099 tiles, and a key range of two top passes."""
    x, form = {"groups_in_place": lambda: (_simplex(24, 1e-10, 13), 0),
               "one_long_group": lambda: (_simplex(20, 1e-12, 12), 2),
               "last_places": lambda: ((np.eye(20) + np.where(np.eye(20), 0, np.random.default_rng(5).random((20, 20)) *
                                                              1e-14)).astype(np.float32), None),
               "many_tiles": lambda: (_two_clusters(1500, 41), 2),
               "two_top_passes": lambda: (_two_pairs(), 0)}[name]()
    if form is None:  # either is right: the group of 190 may or may not be in order
        from paper_2203_02527_gb300 import ph0
        form = ph0.barcodes(torch.from_numpy(x).cuda(), tuning={"packed_sort": 0}).stats["sort_form"]
        assert form in (0, 2)
    run(x, {"packed_sort": 0}, form)


@pytest.mark.parametrize("split,tile,top", [(0, 128, 9), (5, 64, 9), (16, 32, 8), (11, 128, 8), (8, 32, 9)])
def test_settings_with_a_sort(split, tile, top):
    t = {"dist_split16": split, "dist_tile": tile, "sort_top_bits": top, "packed_sort": 0}
    for x in (inputs.noisy_circles(150, 4, 8, seed=91), inputs.with_duplicates(500, 3, 300, seed=92),
              inputs.uniform(300, 37, seed=94)):
        run(x, t, 0)
    run(inputs.exponent_gaps(200, 4, seed=93), t, 2)  # rows whose distances agree in 36 bits


@functools.lru_cache(maxsize=None)
def _far(d):
    x = inputs.uniform(2950 if d < 4 else 4400, d, seed=96 + d)
    x[:, 0] += np.float32(1000.0)
    return x, oracle.barcodes(x)


@pytest.mark.parametrize("split,tile", [(0, 128), (5, 64), (16, 32), (11, 128), (8, 32), (16, 64)])
@pytest.mark.parametrize("d", [2, 5, 33])
def test_settings_without_a_sort(split, tile, d):
    """Above 2,896 points the form without a sort takes the distance kernel's
    settings; coordinates far from zero need more than 32 bits each, their
    differences fewer."""
    from paper_2203_02527_gb300 import ph0
    x, (want, inf_v, nd) = _far(d)
    got = ph0.barcodes(torch.from_numpy(x).cuda(), tuning={"dist_split16": split, "dist_tile": tile})
    assert got.stats["sort_form"] == 3
    assert_bars_equal(got.numpy(), want)
    assert got.inf[0] == inf_v and got.stats["n_distinct"] == nd


def test_served_clouds_that_take_the_short_sort():
    """In the serving context: clouds that sort by default (2,900 to 4,300
    points in four or more dimensions) whose keys do not pack, one of them
    with a group that needs the complete sort, so that it runs again in full."""
    from paper_2203_02527_gb300 import ph0
    from paper_2203_02527_gb300.serve import Server, run_stream
    crowded = _crowded_in(3000, 8, seed=993)
    crowded[1], crowded[2999] = crowded[0], crowded[1500]  # zeros: the keys' top part spans too much to pack
    clouds = [inputs.with_duplicates(2900, 4, 900, seed=97), crowded, inputs.with_duplicates(3700, 8, 50, seed=98)]
    clouds += [inputs.uniform(200 + 31 * i, 3, seed=99 + i) for i in range(5)]
    forms = [ph0.barcodes(torch.from_numpy(x).cuda()).stats["sort_form"] for x in clouds[:3]]
    assert forms == [0, 2, 0]
    with Server(mem_budget=4 << 30, streams=4, small_max_n=180, batch_max=32) as srv:
        done = run_stream(srv, clouds)
    for i, x in enumerate(clouds):
        assert done[i].status == 0
        assert_bars_equal(done[i].bars, oracle.barcodes(x)[0])
