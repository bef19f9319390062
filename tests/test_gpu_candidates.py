"""The candidate path of the threshold kernel where it changes form: sets of candidates around what was once sorted (512) and
what is held at all (2048), spread over the row or gathered in one block's part of it, segments that stay in the
shared-memory ring and segments that do not, ties at the bound, and a first bound that lets too many candidates in.  Oracle and tolerances are those of test_gpu_truncation."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_truncation import check, gpu_threshold, values_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 1 << 12)
    yield c
    c.destroy()


def planted_rows(rng, V, n, bf16, gathered=False, ties=False):
    """Rows whose first n tokens in probability stand far above the rest, nearly equally likely."""
    x = (rng.standard_normal((3, V)) * 0.5 - 40.0).astype(np.float32)
    for row in x:
        at = rng.choice(max(n, V // 16) if gathered else V, size=n, replace=False)
        row[at] = 1.0 if ties else rng.uniform(0.0, 1.0, size=n)
    return W.to_bf16_bits(x) if bf16 else x


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("S,V", [(1, 16000), (1, 40013), (3, 40013), (8, 152064)])
@pytest.mark.parametrize("n", [1, 511, 512, 513, 2047, 2048, 2049])
def test_nucleus_sets_of_every_size(ctx, oracle, S, V, n, bf16):
    import torch
    rng = np.random.default_rng(1000 * S + n)
    T, p, h = 0.9, 0.9, 0.3
    ctx.set_cluster_size(S)
    try:
        for gathered in (False, True):
            rows = planted_rows(rng, V, n, bf16, gathered)
            B = rows.shape[0]
            d_rows, u = tl.to_device(rows), rng.random(B).astype(np.float32)
            thr = torch.zeros(B, device="cuda"); stats = torch.zeros(B, 2, device="cuda")
            tok = torch.zeros(B, dtype=torch.int32, device="cuda"); ent = torch.zeros(B, device="cuda")
            stop = torch.zeros(B, dtype=torch.uint8, device="cuda")
            ctx.draft_step_truncated(d_rows, tl.dtype_code(rows), B, V, V, T, h, 0, p, tl.to_device(u), None, thr, tok, ent,
                                     stop, stats)
            thr2 = torch.zeros(B, device="cuda"); stats2 = torch.zeros(B, 2, device="cuda")
            ctx.row_threshold(d_rows, tl.dtype_code(rows), B, V, V, T, 0, p, thr2, stats2)
            torch.cuda.synchronize()
            t = thr.cpu().numpy()
            assert np.array_equal(t, thr2.cpu().numpy())
            check(oracle, rows, T, 0, p, t, "n=%d S=%d" % (n, S))
            masked = oracle.mask_below(rows, t.astype(np.float64))
            tl.check_draft_against_oracle(oracle, masked, T, h, u, (tok.cpu().numpy(), ent.cpu().numpy(), stop.cpu().numpy(),
                                                                    None), "n=%d S=%d" % (n, S))
            vals = values_of(rows)
            for st in (stats.cpu().numpy(), stats2.cpu().numpy()):
                for b in range(B):
                    Z = np.exp((vals[b][vals[b] >= float(t[b])] - vals[b].max()) / T).sum()
                    # 2^-40 fixed point of 2-ulp exponentials, summed over at most 2049 tokens
                    assert st[b, 0] == np.float32(vals[b].max()) and abs(st[b, 1] - Z) <= 1e-5 * Z
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


@pytest.mark.parametrize("S,V", [(1, 16000), (3, 40013), (8, 152064)])
@pytest.mark.parametrize("n", [64, 513, 2049])
def test_ties_at_the_top_k_bound(ctx, oracle, S, V, n):
    rng = np.random.default_rng(n + S)
    ctx.set_cluster_size(S)
    try:
        for bf16 in (False, True):
            rows = planted_rows(rng, V, n, bf16, ties=True)
            for k, p in ((1, 1.0), (63, 0.9), (64, 1.0), (65, 1.0), (128, 0.9)):
                check(oracle, rows, 1.0, k, p, gpu_threshold(ctx, rows, 1.0, k, p), "S=%d n=%d k=%d" % (S, n, k))
    finally:
        ctx.set_cluster_size(0)


def group_maxima(row, S, per_warp):
    """Maxima of the groups of neighbouring threads from which the first bound of a top-k is taken: the vectors of a warp's segment
    go to its lanes in turn.  fp32 rows that start and end at a vector."""
    vectors = row.reshape(-1, 4).max(axis=1)
    nseg = 16 * S
    vps = ((vectors.size + nseg - 1) // nseg + 7) // 8 * 8
    out = []
    for lo in range(0, vectors.size, vps):
        seg = vectors[lo:lo + vps]
        group = np.arange(seg.size) % 32 * per_warp // 32
        out += [seg[group == j].max() for j in range(per_warp)]
    return np.array(out)


def test_likely_tokens_in_few_groups_of_threads(ctx, oracle):
    # rows that do not fit the ring, their likely tokens all in one warp's segment: most of the group maxima are those of unlikely
    # tokens, the first bound lets in more than the tables hold, and the maxima of stretches have to give a second one
    V, n, k = 152064, 100, 50
    rng = np.random.default_rng(5)
    x = rng.standard_normal((n, V)).astype(np.float32)
    for S, per_warp in ((1, 8), (2, 4)):       # as many groups as have at least 3/2 k
        rows = x.copy()
        segment = V // (16 * S)
        for row in rows[::7]:
            at = int(rng.integers(0, 16 * S)) * segment
            row[at + rng.choice(segment, 2500, replace=False)] += 20.0
            bound = np.sort(group_maxima(row, S, per_warp))[-k]
            assert bound < 10.0 and (row >= bound).sum() > 2048
        ctx.set_cluster_size(S)
        try:
            for p in (1.0, 0.9):
                check(oracle, rows, 1.0, k, p, gpu_threshold(ctx, rows, 1.0, k, p), "S=%d p=%g" % (S, p))
        finally:
            ctx.set_cluster_size(0)
