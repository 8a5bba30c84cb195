"""The serving context when a launch fails after part of a cloud's work was
queued: the cloud is reported as failed, and its device memory goes to no
other cloud before its stream was waited for (csrc/ph0_serve.cu, against a
fake of the CUDA calls: no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2203_02527_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("serve") / "serve_failure_check")
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-cudart", "none",
                           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", exe,
                           os.path.join(HERE, "native", "serve_failure_check.cu"),
                           os.path.join(HERE, "native", "serve_fake_cuda.cpp"), os.path.join(CSRC, "ph0_serve.cu"), "-lpthread"])
    return exe


@pytest.mark.parametrize("which", ["first", "again"])
def test_memory_of_a_failed_launch_waits_for_its_stream(checker, which):
    out = subprocess.run([checker, which], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out
    clouds, failed, overlaps = map(int, out.stdout.split())
    assert (clouds, failed) == (3, 1)
    assert overlaps == 0
