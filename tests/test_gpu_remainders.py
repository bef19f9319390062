"""Segments whose lanes end at every place of the ring: whole rings, remainders of every length, and lanes of one warp that have
one vector more than the others, for the draft step with and without sampling, the row statistics of the verification, and the
thresholds."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_candidate_sets import check_truncated

pytestmark = pytest.mark.gpu

WARPS = 16
COUNTS = (1, 2, 3, 4, 5, 6, 7, 8, 9, 15, 16, 17, 23)       # vectors a lane


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 64)
    yield c
    c.destroy()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("more", [0, 16])
def test_every_remainder(ctx, oracle, more, bf16):
    rng = np.random.default_rng(more + bf16)
    ctx.set_cluster_size(1)
    try:
        for per_lane in COUNTS:
            V = WARPS * (32 * per_lane + more) * (8 if bf16 else 4)
            q = (rng.standard_normal((3, V)) * 2.0).astype(np.float32)
            q[1, -1] = q[2, 0] = 9.0                    # the largest logit at either end
            t = (q + rng.standard_normal((3, V)) * 0.5).astype(np.float32)
            if bf16:
                q, t = W.to_bf16_bits(q), W.to_bf16_bits(t)
            u = rng.random(3).astype(np.float32)
            label = "%d vectors a lane, %d lanes with one more" % (per_lane, more)
            for T in (1.0, 0.0):
                got = tl.gpu_draft_step(ctx, q, T, 0.3, u)
                tl.check_draft_against_oracle(oracle, q, T, 0.3, u, got, label)
                cu = np.array([0, 3])
                tok, uv = got[0][:2].astype(np.int32), u
                if T:
                    uv, _ = tl.guard_accept_uniforms(oracle, tok, q[:2], t, cu, T, u)
                res, early = tl.gpu_verify(ctx, tok, q[:2], t, cu, 2, T, uv, fixed_K=True, early_exit=True)
                tl.check_verify_against_oracle(oracle, tok, q[:2], t, cu, T, uv, res, label)
                tl.check_verify_against_oracle(oracle, tok, q[:2], t, cu, T, uv, early, label)
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("more", [0, 16])
def test_every_remainder_of_the_thresholds(ctx, oracle, more, bf16):
    rng = np.random.default_rng(10 + more + bf16)
    ctx.set_cluster_size(1)
    try:
        for per_lane in COUNTS:
            V = WARPS * (32 * per_lane + more) * (8 if bf16 else 4)
            x = (rng.standard_normal((2, V)) * 0.5 - 30.0).astype(np.float32)
            x[0, rng.choice(V, 80, replace=False)] = rng.uniform(0.0, 4.0, 80)      # spread over the row ...
            for seg in range(0, V, V // WARPS):                                     # ... or at either end of every segment
                x[1, [seg, seg + V // WARPS - 1]] = rng.uniform(0.0, 4.0, 2)
            rows = W.to_bf16_bits(x) if bf16 else x
            u = rng.random(2).astype(np.float32)
            for k, p in ((0, 0.9), (20, 1.0)):
                check_truncated(ctx, oracle, rows, 1.0, k, p, u, "%d vectors a lane, %d lanes with one more, k=%d" % (per_lane, more, k))
        assert ctx.read_status() == 0
    finally:
        ctx.set_cluster_size(0)
