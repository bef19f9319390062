"""Large candidate sets of the threshold kernel: more group maxima than one warp searches (512) and more candidates than
it sorts (256), up to what the tables hold (2048), with and without a nucleus inside the top-k; and that such a call costs a small
multiple of a small top-k and not its square.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_truncation import check, values_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 1 << 12)
    yield c
    c.destroy()


def truncated(ctx, rows, T, k, p, u, h=0.3):
    """Thresholds, statistics and the draft step; the two calls must agree on the thresholds."""
    import torch
    B, V = rows.shape
    d = tl.to_device(rows)
    z = lambda *s, d=torch.float32: torch.zeros(*s, dtype=d, device="cuda")  # noqa: E731
    thr, thr2, stats, stats2, ent = z(B), z(B), z(B, 2), z(B, 2), z(B)
    tok, stop = z(B, d=torch.int32), z(B, d=torch.uint8)
    ctx.draft_step_truncated(d, tl.dtype_code(rows), B, V, V, T, h, k, p, tl.to_device(u), None, thr, tok, ent, stop, stats)
    ctx.row_threshold(d, tl.dtype_code(rows), B, V, V, T, k, p, thr2, stats2)
    torch.cuda.synchronize()
    assert np.array_equal(thr.cpu().numpy(), thr2.cpu().numpy())
    return thr.cpu().numpy(), (stats.cpu().numpy(), stats2.cpu().numpy()), (tok.cpu().numpy(), ent.cpu().numpy(),
                                                                           stop.cpu().numpy(), None)


def check_truncated(ctx, oracle, rows, T, k, p, u, label):
    t, stats, step = truncated(ctx, rows, T, k, p, u)
    check(oracle, rows, T, k, p, t, label)
    tl.check_draft_against_oracle(oracle, oracle.mask_below(rows, t.astype(np.float64)), T, 0.3, u, step, label)
    vals = values_of(rows)
    for st in stats:
        for b, v in enumerate(vals):
            Z = np.exp((v[v >= float(t[b])] - v.max()) / T).sum()
            # 2^-40 fixed point of 2-ulp exponentials over at most 2048 tokens
            assert st[b, 0] == np.float32(v.max()) and abs(st[b, 1] - Z) <= 1e-5 * Z, label


@pytest.mark.parametrize("S", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_every_large_top_k(ctx, oracle, S, bf16):
    rng = np.random.default_rng(S)
    x = (rng.standard_normal((4, 40013)) * np.array([[0.5], [2.0], [4.0], [1.0]])).astype(np.float32)
    x[3, ::5] = x[3, 0]                                    # ties
    rows = W.to_bf16_bits(x) if bf16 else x
    u = np.array([0.0, 1.0 - 2.0 ** -24, 0.5, rng.random()], dtype=np.float32)
    ctx.set_cluster_size(S)
    try:
        for k in (127, 128, 129, 180, 255, 256, 257, 300, 511, 512, 513, 700, 1000, 1024):
            if k <= S * 128:                               # a quarter of the threads of the cluster
                for p in (1.0, 0.9):
                    check_truncated(ctx, oracle, rows, 0.9, k, p, u, "S=%d k=%d p=%g" % (S, k, p))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


def planted(rng, B, V, n, lo=0.0, hi=1.0):
    """n tokens nearly equally likely, far above the rest, all of them in the part [lo, hi) of the row."""
    x = (rng.standard_normal((B, V)) * 0.5 - 40.0).astype(np.float32)
    for row in x:
        row[int(lo * V) + rng.choice(int((hi - lo) * V), n, replace=False)] = rng.uniform(0.0, 1.0, n)
    return x


@pytest.mark.parametrize("S", [2, 3, 4, 6, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_likely_tokens_in_the_part_of_one_block(ctx, oracle, S, bf16):
    # around what a block pushes (2048 / S), what it holds (1024), and with the rest of the table filled by another block
    rng = np.random.default_rng(10 * S)
    V, region = 40013, 2048 // S
    u = rng.random(2).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for n in (region - 1, region, region + 1, 1000, 1023, 1024, 1025):
            for block in (0, 1, S - 1):
                x = planted(rng, 2, V, n, (block + 0.05) / S, (block + 0.9) / S)
                if n >= 1000:
                    other = (block + 1) % S
                    x[1] = np.maximum(x[1], planted(rng, 1, V, 1020, (other + 0.05) / S, (other + 0.9) / S)[0])
                rows = W.to_bf16_bits(x) if bf16 else x
                check_truncated(ctx, oracle, rows, 1.0, 0, 0.9, u, "S=%d n=%d block=%d" % (S, n, block))
                if not bf16 and 300 <= S * 128:
                    check_truncated(ctx, oracle, rows, 1.0, 300, 0.9, u, "k, S=%d n=%d block=%d" % (S, n, block))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


@pytest.mark.parametrize("S", [2, 3, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_nucleus_of_all_the_table_holds_in_the_part_of_one_block(ctx, oracle, S, bf16):
    rng = np.random.default_rng(20 * S)
    V = 40013
    u = rng.random(2).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for n in (1026, 1500, 2047, 2048, 2049):
            for block in (0, S - 1):
                x = planted(rng, 2, V, n, (block + 0.05) / S, (block + 0.9) / S)
                rows = W.to_bf16_bits(x) if bf16 else x
                check_truncated(ctx, oracle, rows, 1.0, 0, 0.9, u, "S=%d n=%d block=%d" % (S, n, block))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


def us_per_call(ctx, rows, k, p, calls=16, replays=9):
    """Median time of a threshold call, from a graph of them."""
    import torch
    B, V = rows.shape
    d = tl.to_device(rows)
    thr, stats = torch.zeros(B, device="cuda"), torch.zeros(B, 2, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx.graph_begin(st)
    for _ in range(calls):
        ctx.row_threshold(d, tl.dtype_code(rows), B, V, V, 1.0, k, p, thr, stats, st)
    g = ctx.graph_end(st)
    times = []
    for _ in range(replays + 2):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(st); g.launch(st); b.record(st); st.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / calls)
    g.destroy()
    return sorted(times[2:])[replays // 2]


@pytest.mark.parametrize("B,V", [(16, 152064), (64, 32000)])
def test_large_sets_do_not_cost_their_square(ctx, B, V):
    # measured on these rows, in times the top-k of 50: large k 1.4 to 1.7, nucleus sets 1.7 to 2.3; by counting, and by a
    # descent with 64-bit atomics, 7 to 25 and 2.7 to 5.5
    x = np.random.default_rng(1).standard_normal((B, V // 2)).astype(np.float32)
    base = us_per_call(ctx, x, 50, 1.0)
    for k in (300, 500) + ((1000,) if V > 100000 else ()):
        assert us_per_call(ctx, x, k, 1.0) < 2.5 * base, k
    for n in (900, 1500):
        rows = W.to_bf16_bits(planted(np.random.default_rng(n), B, V, n))
        assert us_per_call(ctx, rows, 0, 0.9) < 3.2 * base, n


@pytest.mark.parametrize("S", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_vocabulary_in_order_of_frequency(ctx, oracle, S, bf16):
    # all likely tokens lie in the first warps, where the maxima of large groups bound next to nothing
    rng = np.random.default_rng(S)
    x = -1.1 * np.log(np.arange(1, 60002)) + 0.2 * rng.standard_normal((3, 60001))
    x[1] = x[1][::-1]
    rows = W.to_bf16_bits(x.astype(np.float32)) if bf16 else x.astype(np.float32)
    u = rng.random(3).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for k in (1, 7, 50, 100, 128):
            check_truncated(ctx, oracle, rows, 0.8, k, 0.95, u, "S=%d k=%d" % (S, k))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


def test_order_of_frequency_costs_little_more(ctx):
    # measured 2.2 times the shuffled vocabulary; without the second attempt, by the descent over the row, 3.3 to 4.1
    rng = np.random.default_rng(3)
    for B in (1, 16, 64):
        x = (-1.1 * np.log(np.arange(1, 50022)) + 0.2 * rng.standard_normal((B, 50021))).astype(np.float32)
        shuffled = us_per_call(ctx, np.ascontiguousarray(x[:, rng.permutation(50021)]), 50, 1.0)
        assert us_per_call(ctx, x, 50, 1.0) < 2.7 * shuffled, B


@pytest.mark.parametrize("S", [1, 2, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_order_of_frequency_in_the_ring(ctx, oracle, S, bf16):
    # rows that stay in the ring, with one block per row too; k on either side of where a second bound is tried
    rng = np.random.default_rng(30 + S)
    V = 16384 if not bf16 else 30011
    x = -1.1 * np.log(np.arange(1, V + 1)) + 0.2 * rng.standard_normal((3, V))
    x[1] = x[1][::-1]
    rows = W.to_bf16_bits(x.astype(np.float32)) if bf16 else x.astype(np.float32)
    u = rng.random(3).astype(np.float32)
    ctx.set_cluster_size(S)
    try:
        for k in (20, 50, 100, 128, 129, 300, 1000):
            if k <= S * 128:
                check_truncated(ctx, oracle, rows, 0.8, k, 0.95, u, "S=%d k=%d" % (S, k))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


def test_order_of_frequency_does_not_pay_for_attempts_that_fail(ctx):
    # one block per row, in the ring: measured 1.5 times the shuffled vocabulary; with a bound from the threads' maxima first, which
    # here is no better than the first one, 3.6
    rng = np.random.default_rng(9)
    V = 32000
    x = (-1.1 * np.log(np.arange(1, V + 1)) + 0.2 * rng.standard_normal((600, V))).astype(np.float32)
    shuffled = us_per_call(ctx, W.to_bf16_bits(np.ascontiguousarray(x[:, rng.permutation(V)])), 100, 0.9)
    assert us_per_call(ctx, W.to_bf16_bits(x), 100, 0.9) < 2.2 * shuffled
    # a large k: measured 1.45 times one so large that the row goes to the descent at once; with a second bound tried first 2.05
    rows = W.to_bf16_bits(x[:64])
    assert us_per_call(ctx, rows, 300, 1.0) < 1.75 * us_per_call(ctx, rows, 1000, 1.0)


def test_gathered_sets_cost_what_spread_ones_do(ctx):
    # measured: 1.1 to 1.2 times; where the candidates of a block did not fit the table and the row took the descent 1.5 to 1.6
    rng = np.random.default_rng(2)
    for B, V, n in ((16, 152064, 700), (1, 152064, 400)):
        spread = us_per_call(ctx, W.to_bf16_bits(planted(rng, B, V, n)), 0, 0.9)
        assert us_per_call(ctx, W.to_bf16_bits(planted(rng, B, V, n, 0.0, 0.1)), 0, 0.9) < 1.35 * spread, (B, V, n)


def test_gathered_sets_of_many_rows_cost_what_spread_ones_do(ctx):
    # long rows, somewhat more than SMs, three blocks each.  Measured 0.95 to 1.0 times; with room for 1024 candidates of a block, where
    # the row took the descent, 2.1 to 2.3
    rng = np.random.default_rng(6)
    for B, V, n in ((160, 152064, 1500), (152, 200000, 1900)):
        spread = us_per_call(ctx, W.to_bf16_bits(planted(rng, B, V, n)), 0, 0.9)
        assert us_per_call(ctx, W.to_bf16_bits(planted(rng, B, V, n, 0.0, 0.1)), 0, 0.9) < 1.35 * spread, (B, V, n)


def test_flat_rows_leave_the_candidates_soon(ctx):
    # a nucleus of tens of thousands of tokens takes the descent by mass; with a top-k that drops nothing but one token the
    # row takes the same descent after one by counts.  Measured 0.92 of that; collecting to the end 1.1
    rng = np.random.default_rng(4)
    for B, V in ((300, 32000), (16, 152064)):
        x = -1.1 * np.log(np.arange(1, V + 1))
        rows = W.to_bf16_bits(np.stack([x[rng.permutation(V)] for _ in range(B)]).astype(np.float32))
        assert us_per_call(ctx, rows, 0, 0.95) < 1.02 * us_per_call(ctx, rows, V - 1, 0.95), (B, V)


def test_flat_rows_are_cut_no_worse_than_by_the_other_kernels(ctx):
    # long rows between 4/3 and 2 per SM.  Measured 1.0 to 1.06 times the best of one and two blocks per row; with three 1.3
    rng = np.random.default_rng(8)
    rows = rng.standard_normal((280, 200000), dtype=np.float32)
    chosen = us_per_call(ctx, rows, 0, 0.95, calls=4)
    best = []
    try:
        for S in (1, 2):
            ctx.set_cluster_size(S)
            best.append(us_per_call(ctx, rows, 0, 0.95, calls=4))
    finally:
        ctx.set_cluster_size(0)
    assert chosen < 1.15 * min(best), (chosen, best)
