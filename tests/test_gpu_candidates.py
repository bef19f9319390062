"""The candidate path of the threshold kernel where it changes form: sets of candidates around what is sorted (512) and
what is held at all (2048), spread over the row or gathered in one block's part of it, segments that stay in the
shared-memory ring and segments that do not, ties at the bound, and a bound from half of the row that lets too many
candidates in.  Oracle and tolerances are those of test_gpu_truncation."""
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


def test_bound_from_half_of_the_row_lets_too_many_in(ctx, oracle):
    # more than 48 MB of logits: the bound comes from the first half of every segment, where this row has nothing
    V, n = 152064, 100
    rng = np.random.default_rng(5)
    x = rng.standard_normal((n, V)).astype(np.float32)
    x[::7] -= 20.0
    for S in (1, 2):
        rows = x.copy()
        nseg = 16 * S
        vps = ((V // 4 + nseg - 1) // nseg + 7) // 8 * 8
        first = np.zeros(V, dtype=bool)
        for seg in range(nseg):
            lo = seg * vps * 4
            first[lo:min(lo + vps * 2, V)] = True
            rows[::7, lo + vps * 2:min(lo + vps * 4, V)] += 20.0 / 2
        for row in rows[::7]:      # what the first half bounds from below does not fit the tables (2048), so there is a second bound
            assert (row >= np.sort(row[first])[-50]).sum() > 2048
        ctx.set_cluster_size(S)
        try:
            for k, p in ((50, 1.0), (50, 0.9)):
                check(oracle, rows, 1.0, k, p, gpu_threshold(ctx, rows, 1.0, k, p), "S=%d k=%d p=%g" % (S, k, p))
        finally:
            ctx.set_cluster_size(0)
