"""Clouds whose distances repeat thousands of times, on the whole path without
a sort, against the oracle bit for bit (positions, indices and keys are
integers, so there is no tolerance): strips of the distance kernel that hold
few distances, and a hash bucket that outgrows its room although no strip
crowds it (and now and then one does)."""
import numpy as np
import pytest

from paper_2203_02527_gb300 import inputs
from tests.test_gpu_direct import check

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _simplex_among_uniform():
    # 100 points at equal distances (4,950 pairs) spread evenly over 1,000:
    # their bucket gets 4,950 + 4,095 keys for a room of 7,230, about 10 + 8
    # in a strip of 1,024 where 26 would crowd it
    x = np.random.default_rng(51).random((1000, 100)).astype(np.float32)
    x[::10] = 0.0
    x[np.arange(0, 1000, 10), np.arange(100)] = 1.0
    return x


@pytest.mark.parametrize("name", ["lattice_14_14_14", "lattice_53_53", "integers_line", "integers_plane", "bytes_16",
                                  "one_point", "simplex_among_uniform"])
def test_repeated_distances(name):
    rng = np.random.default_rng(50)
    x = {"lattice_14_14_14": lambda: inputs.lattice(14, 3),
         "lattice_53_53": lambda: inputs.lattice(53, 2),
         "integers_line": lambda: rng.integers(0, 2896, (2896, 1)).astype(np.float32),
         "integers_plane": lambda: rng.integers(0, 100, (2500, 2)).astype(np.float32),
         "bytes_16": lambda: rng.integers(0, 256, (1500, 16)).astype(np.float32),
         "one_point": lambda: np.full((2896, 3), 0.25, np.float32),
         "simplex_among_uniform": _simplex_among_uniform}[name]()
    check(x)
