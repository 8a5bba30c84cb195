"""The 32-bit squares of the distance kernels under the rule that the kernels
use (coordinates less than 2^32 units apart, wherever they lie), compiled for
the host, against the host's own binary64 arithmetic: the square alone up to
factors of 2^32 - 1, whole distances in 1 to 70 dimensions in every form, and
the rule at its bounds.  Exact equality of the bit patterns is required."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("emu") / "emu64_narrow_check")
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-o", exe,
                           os.path.join(HERE, "native", "emu64_narrow_check.cpp")])
    return exe


@pytest.mark.parametrize("what,count,least", [("squares", 2_000_000, 2_000_000), ("tiles", 7000, 500_000),
                                              ("bounds", 20000, 20000)])
def test_narrow_rule_bit_exact(checker, what, count, least):
    out = subprocess.run([checker, what, "21", str(count)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    checked, bad, narrow, far = map(int, out.stdout.split())
    assert bad == 0 and checked >= least
    if what == "tiles":  # dimensions beyond 32 bits whose differences are not
        assert narrow > 10000 and far > 1000
