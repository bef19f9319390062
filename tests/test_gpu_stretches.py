"""Top-k of rows that do not fit the ring: the candidates come from the stretches of vectors whose maximum reaches the bound.
Row lengths around the edges of a stretch, of the ring and of the table of stretches (more than eight rounds of the ring per
thread: stretches of several rounds), at several phases; and logits that are large against their spread, of which half a key
does not tell one stretch from another.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_candidate_sets import check_truncated, truncated, us_per_call
from test_gpu_truncation import check

pytestmark = pytest.mark.gpu

BLOCK = 16 * 32 * 8       # vectors that fill the ring of a block


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 1 << 12)
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


@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("offset,spread", [(601.0, 3.0), (1200.0, 4.0), (-900.0, 4.0), (20.0, 0.01)])
def test_large_against_their_spread(ctx, oracle, S, offset, spread):
    rng = np.random.default_rng(S)
    x = (offset + spread * rng.standard_normal((3, 256000))).astype(np.float32)
    u = rng.random(3).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for k, p in ((1, 1.0), (50, 1.0), (50, 0.9), (100, 0.9)):
            label = "S=%d %g +- %g, k=%d p=%g" % (S, offset, spread, k, p)
            t, stats, step = truncated(ctx, x, 1.0, k, p, u)
            check(oracle, x, 1.0, k, p, t, label)
            tl.check_draft_against_oracle(oracle, oracle.mask_below(x, t.astype(np.float64)), 1.0, 0.3, u, step, label)
            for st in stats:
                for b, v in enumerate(x.astype(np.float64)):
                    Z = np.exp(v[v >= float(t[b])] - v.max()).sum()
                    # as check_truncated, and the rounding of the largest logit in log2 units, half an ulp of it
                    tol = 1e-5 + np.spacing(np.float32(abs(v.max()) * 1.4427)) / 2 * 0.6932
                    assert st[b, 0] == np.float32(v.max()) and abs(st[b, 1] - Z) <= tol * Z, label
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


def test_large_against_their_spread_costs_little_more(ctx):
    # measured 1.07 and 1.10 times the rows around zero; with a list too short for the stretches that half a key lets through, and
    # candidates taken from it that nothing had written, 16
    rng = np.random.default_rng(7)
    g = rng.standard_normal((64, 256000)).astype(np.float32)
    base = us_per_call(ctx, 4.0 * g, 50, 0.9)
    for offset, spread in ((1200.0, 4.0), (20.0, 0.01)):
        assert us_per_call(ctx, (offset + spread * g).astype(np.float32), 50, 0.9) < 1.5 * base, (offset, spread)
