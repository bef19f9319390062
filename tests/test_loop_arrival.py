"""The counter on which the draft kernel of a recorded drafting loop decides the loop (no GPU: the decision is a host function
too).  The loop ends when the sequences are done or the iterations are used up, and it ends whatever the counter held when it
was entered."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def loop(tmp_path_factory):
    from paper_2411_18462_b200 import build
    exe = str(tmp_path_factory.mktemp("loop") / "harness")
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.INCLUDE, "-I",
                           build.CSRC, "-o", exe, os.path.join(HERE, "loop_arrival_harness.cu")])

    def run(leftover, B, lasts, max_iters):
        out = subprocess.run([exe, str(leftover), str(B), str(lasts), str(max_iters), "1000"], capture_output=True, text=True)
        assert out.returncode == 0
        return tuple(int(x) for x in out.stdout.split())
    return run


@pytest.mark.parametrize("B", [1, 2, 7, 300])
def test_clean_counter(loop, B):
    assert loop(0, B, 1, 9) == (1, 0)
    assert loop(0, B, 5, 9) == (5, 0)
    assert loop(0, B, 50, 9) == (9, 0)


@pytest.mark.parametrize("B", [1, 2, 7, 300])
def test_ends_whatever_the_counter_holds(loop, B):
    for left in (1, B - 1, B, B + 1, 3 * B, (5 << 32) + B, 0xfffffff0):
        body, overrun = loop(left, B, 1000, 9)
        assert body <= 10, (left, body)
        if left >= B:
            assert overrun == 1
    # left-over arrivals that do not fill the batch: the iterations shift, the limit holds
    if B > 1:
        assert loop(B - 1, B, 1000, 9)[0] <= 10
