"""The distance kernel's tile edge in high dimensions, counted by the tiles a
cloud is cut into: 128, 64 and 32 points where two blocks of binary64
coordinates and five words a dimension fit 160 KB, else 16 where they fit 168,
else 8.  The bars are the oracle's."""
import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,edge", [(79, 128), (80, 64), (156, 64), (157, 32), (307, 32), (308, 16), (593, 16), (594, 16),
                                    (610, 16), (623, 16), (624, 8), (1024, 8)])
def test_tile_edge(d, edge):
    from paper_2203_02527_gb300 import ph0
    n = 700
    x = inputs.uniform(n, d, seed=95)
    got = ph0.barcodes(torch.from_numpy(x).cuda(), tuning={"packed_sort": 0})
    side = -(-n // edge)
    assert got.stats["dist_tiles"] == side * (side + 1) // 2
    assert_bars_equal(got.numpy(), oracle.barcodes(x)[0])
