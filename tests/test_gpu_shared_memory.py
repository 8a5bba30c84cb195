"""Kernels whose dynamic shared memory grows with the cloud: their limit holds
for the whole process, so it must suffice for every size whatever ran before
and whatever another thread runs.  The results are the oracle's bit for bit
(positions, indices and keys are integers, so there is no tolerance)."""
import os
import subprocess
import sys
import threading

import pytest

import oracle
from paper_2203_02527_gb300 import inputs
from tests.test_gpu_parity import assert_bars_equal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FRESH = """
import numpy as np, torch, oracle
from paper_2203_02527_gb300 import inputs, ph0
for n in (2450, 2451, 2457, 2458):
    x = inputs.uniform(n, 2, seed=4000 + n)
    got = ph0.barcodes(torch.from_numpy(x).cuda())
    want = oracle.barcodes(x)[0]
    assert got.numpy().tobytes() == want.astype(got.numpy().dtype).tobytes(), n
    assert got.stats["sort_form"] == 3
print("all equal")
"""


def test_counts_around_48_kb_in_a_fresh_process():
    """2,451 to 2,457 points need more than 48 KB less the static part, and
    no more than 48 KB, of the count kernel's dynamic shared memory."""
    out = subprocess.run([sys.executable, "-c", FRESH], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and "all equal" in out.stdout, out.stderr[-2000:]


def queue_side_by_side(clouds, rounds=40, each=128, tuning=None):
    """A thread per cloud, each queueing `each` calls on it by one call of
    ph0_barcodes_many, `rounds` times; what went wrong."""
    import ctypes

    from paper_2203_02527_gb300 import _lib, ph0
    lib, failed, t = _lib.load(), [], _lib.Tuning.make(**tuning) if tuning else None

    def work(x):
        torch.cuda.set_device(0)
        n, d = x.shape
        pts, ws = torch.from_numpy(x).cuda(), ph0.Workspace(n, d)
        raw = torch.empty((n - 1, _lib.BAR_BYTES), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        calls = (_lib.Cloud * each)()
        for c in calls:
            c.pts_dev, c.n, c.ld, c.d, c.bars_dev = pts.data_ptr(), n, d, d, raw.data_ptr()
            c.ws, c.ws_bytes = ws.buf.data_ptr(), ws.nbytes
            if t is not None:
                c.tuning = ctypes.pointer(t)
        handles = (ctypes.c_void_p * 1)(stream.cuda_stream)
        for _ in range(rounds):
            rc = lib.ph0_barcodes_many(calls, each, handles, 1)
            stream.synchronize()
            if rc != 0:
                failed.append((n, rc))
                return
        got = raw.cpu().numpy().reshape(-1).view(_lib.BAR_DTYPE)
        try:
            assert_bars_equal(got, oracle.barcodes(x)[0])
        except AssertionError as e:
            failed.append((n, str(e)))

    threads = [threading.Thread(target=work, args=(x,)) for x in clouds]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    return failed


def test_counts_of_two_sizes_in_two_threads():
    """A thread with 2,896 points and one with 2,500: neither's launches are refused."""
    assert queue_side_by_side([inputs.uniform(n, 2, seed=4100 + n) for n in (2896, 2500)]) == []


def test_reductions_of_two_sizes_in_two_threads():
    """The reduction after a sort, of 300 points and of 2,800: neither's
    launches are refused."""
    clouds = [inputs.uniform(n, 2, seed=4200 + n) for n in (2800, 300)]
    assert queue_side_by_side(clouds, rounds=20, each=64, tuning={"packed_sort": 0}) == []

