"""First homology's least workspace (host arithmetic, no GPU): what one column
in sorted runs needs, or as many bit sets as can be used where those take
less; the best one holds up to 2 GiB of bit sets up to 1024 points."""
import pytest

from paper_2203_02527_gb300 import build, _lib

# bytes that served before columns were reduced as bit sets, in 3 dimensions
RUNS = {128: 34062848, 256: 270084352, 700: 706033152, 1000: 742259456, 1024: 745712640}


@pytest.fixture(scope="module")
def lib():
    build.build()
    return _lib.load()


@pytest.mark.parametrize("n", sorted(RUNS))
def test_what_served_before_serves(lib, n):
    assert lib.ph0_h1_workspace_bytes(n, 3) <= RUNS[n]


def test_least_and_best(lib):
    for n in [*range(1, 300), 400, 511, 512, 700, 900, 1023, 1024, 1025, 2000, 4096]:
        least, best = lib.ph0_h1_workspace_bytes(n, 3), lib.ph0_h1_workspace_best_bytes(n, 3)
        assert 0 < least <= best
        if n > 1024:
            assert least == best
    for n, d in ((0, 3), (4097, 3), (10, 0), (10, 1025)):
        assert lib.ph0_h1_workspace_bytes(n, d) == lib.ph0_h1_workspace_best_bytes(n, d) == 0
