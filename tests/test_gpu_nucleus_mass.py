"""The cut of a nucleus alone does not depend on how many blocks share the row nor on the way the row goes: masses are sums of
integers.  Cuts in dense tails and top_p close to 1, where a total formed in fp32 decides differently from one launch shape
to the next; against fp64 within the 1e-6 that svip.h states."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_truncation import gpu_threshold, values_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 1 << 12)
    yield c
    c.destroy()


def rows_of(rng, kind, V, n=96):
    if kind == "bulk":                 # small enough that every token may be a candidate
        x = rng.standard_normal((n, V)) * rng.uniform(0.5, 3.0, (n, 1))
    else:                              # a few hundred likely tokens above a bulk that carries nothing
        x = rng.standard_normal((n, V)) * 0.5 - 60.0
        for row in x:
            m = int(rng.integers(100, 350))
            row[rng.choice(V, m, replace=False)] = rng.uniform(-4.0, 4.0) - rng.uniform(0.0, 12.0, m)
    x[:, 0] = -np.inf                  # the least likely token has no mass at all
    return x.astype(np.float32)


@pytest.mark.parametrize("kind,V,T", [("bulk", 900, 1.0), ("bulk", 1801, 0.7), ("set", 33001, 1.0), ("set", 152064, 1.0)])
@pytest.mark.parametrize("bf16", [False, True])
def test_same_cut_for_every_launch_shape_and_path(ctx, kind, V, T, bf16):
    rng = np.random.default_rng(V)
    x = rows_of(rng, kind, V)
    rows = W.to_bf16_bits(x) if bf16 else x
    vals = values_of(rows)
    for p in (0.5, 0.9, 0.99, 0.9999, 0.99999):
        # top_k one below the vocabulary drops the token without mass only and takes the radix descent
        want = gpu_threshold(ctx, rows, T, V - 1, p)
        for S in range(1, 9):
            ctx.set_cluster_size(S)
            try:
                got = gpu_threshold(ctx, rows, T, 0, p)
            finally:
                ctx.set_cluster_size(0)
            assert np.array_equal(got, want), (kind, V, p, S, int((got != want).sum()))
        for v, tau in zip(vals, want):
            w = np.exp((v - v.max()) / T)
            assert w[v >= tau].sum() >= (p - 1e-6) * w.sum() and w[v > tau].sum() < (p + 1e-6) * w.sum()
    assert ctx.read_status() == 0
