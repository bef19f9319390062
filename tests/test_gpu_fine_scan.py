"""The fine scan by itself, on weights given as tables: the element whose running sum first exceeds the target, and, where a
run of vectors has a sum at rounding level but no element of its own does (the two are formed by different expressions), an
element with weight all the same."""
import ctypes as C
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def scan(tmp_path_factory):
    import subprocess
    import torch
    from paper_2411_18462_b200 import build
    so = str(tmp_path_factory.mktemp("scan") / "harness.so")
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                           "-fPIC", "-I", build.INCLUDE, "-I", build.CSRC, "-o", so, os.path.join(HERE, "fine_scan_harness.cu")])
    lib = C.CDLL(so)
    lib.scan.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_int, C.c_float, C.c_void_p]

    def run(sums, single, v_lo, v_hi, target):
        a, b = torch.from_numpy(sums).cuda(), torch.from_numpy(single).cuda()
        out = torch.full((1,), -7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.scan(a.data_ptr(), b.data_ptr(), v_lo, v_hi, target, out.data_ptr()) == 0
        return int(out.item())
    return run


# one run of one vector per thread, runs of four, and several rounds of the block
@pytest.mark.parametrize("nv", [1, 33, 512, 700, 2049, 5000])
def test_first_element_above_the_target(scan, nv):
    rng = np.random.default_rng(nv)
    w = np.where(rng.random(4 * nv) < 0.05, rng.integers(1, 9, 4 * nv), 0).astype(np.float32)      # exact sums
    w[-1] = 1.0
    cum = np.cumsum(w)
    for target in (0.0, float(cum[-1]) - 0.5, float(np.floor(cum[-1] * rng.random()))):
        assert scan(w, w, 0, nv, target) == int(np.argmax(cum > target)), target


@pytest.mark.parametrize("nv,at", [(40, 17), (512, 300), (2049, 1030), (5000, 3000)])
def test_run_without_an_element_of_its_own(scan, nv, at):
    # all the mass is noise in one vector, which the look at single elements does not see
    sums = np.zeros(4 * nv, dtype=np.float32)
    sums[4 * at + 1:4 * at + 3] = 2.0 ** -30
    assert scan(sums, np.zeros_like(sums), 0, nv, 2.0 ** -31) == 4 * at + 2
    # the same behind elements that are below the target
    sums[4 * (at // 2)] = 2.0 ** -31
    single = np.where(np.arange(4 * nv) < 4 * at, sums, 0).astype(np.float32)
    assert scan(sums, single, 0, nv, 2.0 ** -30) in (4 * at + 2, 4 * (at // 2))
