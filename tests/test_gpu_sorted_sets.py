"""Candidate sets that one warp sorts: sizes around what it holds two, four and eight of per lane (64, 128, 256) and above, equal
keys across the cut, rows without finite mass.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

from paper_2411_18462_b200 import workloads as W
from test_gpu_candidate_sets import check_truncated

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 64)
    yield c
    c.destroy()


@pytest.mark.parametrize("S", [1, 4])
@pytest.mark.parametrize("bf16", [False, True])
def test_sizes_of_sorted_sets(ctx, oracle, S, bf16):
    # the likely tokens stand apart, so the set has exactly n members; every third row has its members equal in pairs
    rng = np.random.default_rng(S)
    V = 20011
    ctx.set_cluster_size(S)
    try:
        for n in (1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257):
            x = (rng.standard_normal((3, V)) * 0.5 - 60.0).astype(np.float32)
            for b in range(3):
                v = rng.uniform(0.0, 4.0, n)
                x[b, rng.choice(V, n, replace=False)] = np.repeat(v, 2)[:n] if b == 2 else v
            rows = W.to_bf16_bits(x) if bf16 else x
            u = np.array([0.0, 1.0 - 2.0 ** -24, rng.random()], dtype=np.float32)
            for p in (0.9, 0.99999):
                check_truncated(ctx, oracle, rows, 1.0, 0, p, u, "nucleus S=%d n=%d p=%g" % (S, n, p))
            if n <= 128:
                check_truncated(ctx, oracle, rows, 1.0, n, 0.9, u, "top-k S=%d n=%d" % (S, n))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)
