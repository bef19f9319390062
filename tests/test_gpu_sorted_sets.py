"""Candidate sets that one warp sorts: sizes around what it holds two, four and eight of per lane (64, 128, 256) and above, equal
keys across the cut, rows without finite mass.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_candidate_sets import check_truncated, truncated
from test_gpu_truncation import check

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


def far_from_zero(bf16):
    """A logit whose product with log2(e) is rounded by nearly 16, half a unit in the last place, and that error."""
    c = np.float64(np.float32(1.4426950408889634))
    x = np.arange(1.9e8, 3.7e8, 1e6 if bf16 else 1e3).astype(np.float32)
    if bf16:
        x = np.unique(W.bf16_bits_to_f32(W.to_bf16_bits(x)))
    exact = x.astype(np.float64) * c                       # 48 bits: exact
    error = exact - exact.astype(np.float32).astype(np.float64)
    best = int(np.argmax(error))
    return x[best], error[best]


@pytest.mark.parametrize("S", [1, 4])
@pytest.mark.parametrize("bf16", [False, True])
def test_logits_far_from_zero(ctx, S, bf16):
    # the mass of the largest logit is 2^40 times 2 to the rounding error of its product with log2(e): four of them make about 2^58
    x, error = far_from_zero(bf16)
    assert error > 14.5
    V, n = 3001, 4
    at = np.array([5, 700, 1501, 2999])
    v = np.full((8, V), x - np.float32(6.4e7), dtype=np.float32)
    v[:, at] = x
    rows = W.to_bf16_bits(v) if bf16 else v
    u = ((np.arange(8) + 0.5) / 8).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for k, p in ((4, 1.0), (4, 0.9), (0, 0.9)):
            thr, stats, (tok, ent, _, _) = truncated(ctx, rows, 1.0, k, p, u)
            label = "S=%d k=%d p=%g" % (S, k, p)
            assert np.all(thr == x), label
            assert np.array_equal(tok, at[np.floor(u * n).astype(int)]), (label, tok)
            # ln 4 from terms of the size of the error in log2 units, each of 2-ulp exponentials
            assert np.all(np.abs(ent - np.log(n)) <= 1e-4), (label, ent)
            for st in stats:
                assert np.all(st[:, 0] == x) and np.all(np.abs(st[:, 1] / (n * 2.0 ** error) - 1.0) <= 1e-5), (label, st)
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


@pytest.mark.parametrize("S", [1, 4])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("V", [200, 20011])
def test_rows_without_finite_mass(ctx, oracle, V, bf16, S):
    # their draft step is streamed at the threshold by the whole cluster, after block 0 has sorted the candidates: the same results as
    # from the two separate calls, next to rows that are finished from their candidates.  With the short rows every token is a candidate
    import torch
    rng = np.random.default_rng(V + S)
    x = (rng.standard_normal((7, V)) * 2.0).astype(np.float32)
    x[1] = -np.inf
    x[2, V // 3] = np.inf
    x[3, V // 2] = 2.0e29                 # beyond what counts as finite
    x[4] = np.nan
    x[5] = -2.0e29
    finite = [0, 6]
    rows = W.to_bf16_bits(x) if bf16 else x
    u = rng.random(7).astype(np.float32)
    d, dt = tl.to_device(rows), tl.dtype_code(rows)
    ctx.set_cluster_size(S)
    try:
        for k, p in ((50, 1.0), (50, 0.9), (1, 1.0), (0, 0.9)):
            label = "V=%d S=%d k=%d p=%g" % (V, S, k, p)
            ctx.read_status()
            thr, stats, step = truncated(ctx, rows, 1.0, k, p, u)
            assert ctx.read_status() == 1, label        # a row without finite mass, and nothing else
            z = lambda *s, d=torch.float32: torch.zeros(*s, dtype=d, device="cuda")  # noqa: E731
            st, tok, ent, stop = z(7, 2), z(7, d=torch.int32), z(7), z(7, d=torch.uint8)
            ctx.draft_step_filtered(d, dt, 7, V, V, 1.0, 0.3, tl.to_device(u), None, tl.to_device(thr), tok, ent, stop, st)
            torch.cuda.synchronize()
            other = [b for b in range(7) if b not in finite]
            for got, want in zip((step[0], step[1], step[2], stats[0]), (tok, ent, stop, st)):
                assert np.array_equal(got[other], want.cpu().numpy()[other], equal_nan=got.dtype == np.float32), label
            check(oracle, rows[finite], 1.0, k, p, thr[finite], label)
            tl.check_draft_against_oracle(oracle, oracle.mask_below(rows[finite], thr[finite].astype(np.float64)), 1.0, 0.3, u[finite],
                                          tuple(a[finite] for a in step[:3]) + (None,), label)
    finally:
        ctx.set_cluster_size(0)
