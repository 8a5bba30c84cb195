"""First homology in workspaces between the least and the best: the same bars
bit for bit (integers and keys, so there is no tolerance) whether the columns
are reduced as many, a few or no bit sets at a time; one byte less is refused;
and ph0.h1 uses the least when the best cannot be allocated."""
import ctypes

import numpy as np
import pytest

from paper_2203_02527_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(3, 2), (60, 3), (130, 2), (300, 8), (520, 2), (700, 2), (1024, 2)])
def test_any_room_gives_the_same_bars(n, d):
    from paper_2203_02527_gb300 import _lib, ph0
    lib = _lib.load()
    x = torch.from_numpy(inputs.uniform(n, d, seed=4400 + n)).cuda()
    want, _ = ph0.h1(x)
    m = n * (n - 1) // 2
    least, best = int(lib.ph0_h1_workspace_bytes(n, d)), int(lib.ph0_h1_workspace_best_bytes(n, d))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for room in (least, least + (best - least) // 9, (least + best) // 2):
        bars = torch.zeros((m - (n - 1), _lib.H1_BAR_BYTES), dtype=torch.uint8, device="cuda")
        guard = torch.full((room + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
        assert lib.ph0_h1(x.data_ptr(), n, d, d, bars.data_ptr(), guard.data_ptr(), room, stream, None) == 0
        assert bars.cpu().numpy().tobytes() == want.tobytes()
        assert bool((guard[room:] == 0xA5).all())
        del guard
    ws = torch.empty(least, dtype=torch.uint8, device="cuda")
    assert lib.ph0_h1(x.data_ptr(), n, d, d, bars.data_ptr(), ws.data_ptr(), least - 1, stream, None) == 4


def test_h1_without_memory_for_the_best():
    from paper_2203_02527_gb300 import ph0
    x = torch.from_numpy(inputs.uniform(700, 2, seed=4500)).cuda()
    want, _ = ph0.h1(x)
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + 1.5e9) / total)
    try:
        got, _ = ph0.h1(x)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert np.array_equal(got, want)
