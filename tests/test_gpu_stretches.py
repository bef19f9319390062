"""Top-k of rows that do not fit the ring: the candidates come from the stretches of vectors whose maximum reaches the bound.
Row lengths around the edges of a stretch, of the ring and of the table of stretches (more than eight rounds of the ring per
thread: stretches of several rounds), at several phases.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

from paper_2411_18462_b200 import workloads as W
from test_gpu_candidate_sets import check_truncated

pytestmark = pytest.mark.gpu

BLOCK = 16 * 32 * 8       # vectors that fill the ring of a block


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 64)
    yield c
    c.destroy()


@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("rings", [1, 2, 8, 9])
@pytest.mark.parametrize("bf16", [False, True])
def test_edges_of_stretches(ctx, oracle, S, rings, bf16):
    rng = np.random.default_rng(rings + 100 * S)
    per_vector = 8 if bf16 else 4
    ctx.set_cluster_size(S)
    try:
        for extra in (-16, 1, 128 * per_vector + 3):
            V = rings * BLOCK * S * per_vector + extra
            x = (rng.standard_normal((3, V)) * 2.0).astype(np.float32)
            x[0, -40:] += 20.0                                   # likely tokens gathered at the end of the row ...
            x[1, rng.integers(0, V, 60)] += 15.0                 # ... spread over it ...
            x[2] = np.sort(x[2])[::-1]                           # ... and all logits in descending order
            rows = W.to_bf16_bits(x) if bf16 else x
            for k in (1, 50):
                check_truncated(ctx, oracle, rows, 1.0, k, 0.9, rng.random(3).astype(np.float32), "S=%d V=%d k=%d" % (S, V, k))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)
