"""Kernels whose dynamic shared memory grows with the cloud: their limit holds
for the whole process, so it must suffice for every size whatever ran before
and whatever another thread runs.  The results are the oracle's bit for bit
(positions, indices and keys are integers, so there is no tolerance)."""
import os
import subprocess
import sys
import threading

import numpy as np
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


def run_side_by_side(sizes, call, rounds):
    """call(x) for each size in a thread of its own; the exceptions."""
    failed = []

    def work(n):
        try:
            torch.cuda.set_device(0)
            x = torch.from_numpy(inputs.uniform(n, 2, seed=4100 + n)).cuda()
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds):
                    call(x)
        except Exception as e:  # noqa: BLE001
            failed.append((n, repr(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return failed


def test_counts_of_two_sizes_in_two_threads():
    """A thread with 2,896 points and one with 2,500: neither's launches are
    refused, and the bars stay right."""
    from paper_2203_02527_gb300 import ph0
    ws = {n: ph0.Workspace(n, 2) for n in (2500, 2896)}
    want = {n: oracle.barcodes(inputs.uniform(n, 2, seed=4100 + n))[0] for n in ws}

    def call(x):
        got = ph0.barcodes(x, ws[len(x)])
        if not np.array_equal(got.numpy()["order"], want[len(x)]["order"]):
            raise AssertionError("order")

    assert run_side_by_side(list(ws), call, 300) == []
    for n in ws:
        x = torch.from_numpy(inputs.uniform(n, 2, seed=4100 + n)).cuda()
        assert_bars_equal(ph0.barcodes(x, ws[n]).numpy(), want[n])
