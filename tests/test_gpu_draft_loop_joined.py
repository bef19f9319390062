"""A drafting loop whose policy step is taken by the draft kernel gives what the loop with a policy kernel of its own gives
(anything recorded between the two calls keeps them apart): batches of one and several blocks per row, sampling and
greedy, all sequences finishing together or one by one, and more iterations than any sequence needs."""
import numpy as np
import pytest

import svip_testlib as tl
from paper_2411_18462_b200 import workloads as W
from test_gpu_draft_loop import make_bufs, pools

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2411_18462_b200 import Context
    c = Context(0, 4096)
    yield c
    c.destroy()


@pytest.mark.parametrize("B,V", [(1, 32000), (5, 2048), (300, 1000)])
@pytest.mark.parametrize("T", [1.0, 0.0])
@pytest.mark.parametrize("policy,max_iters", [(0, 9), (1, 9), (2, 3)])
def test_joined_and_separate_policy_step_agree(ctx, B, V, T, policy, max_iters):
    import torch
    w = W.make_workload("ragged", B=B, V=V, K_max=6)
    K_cap = w.K_max
    q_pm, _ = pools(w)
    rng = np.random.default_rng(B)
    gamma = rng.integers(1, K_cap + 1, B).tolist()
    ud = torch.from_numpy(rng.random(K_cap * B).astype(np.float32)).cuda()
    got = []
    for apart in (False, True):
        bufs = make_bufs(torch, q_pm, B, K_cap, gamma)
        bufs["ud"].copy_(ud)
        bufs["act"][B // 2:B // 2 + 1] = 1 if B == 1 else 0        # one sequence is not drafting
        torch.cuda.synchronize()
        st = torch.cuda.Stream()
        before = ctx.launch_count()
        ctx.graph_begin(st)
        body = ctx.graph_loop_begin(st, bufs["nact"], max_iters)
        ctx.draft_step_at(bufs["q"], tl.dtype_code(w.q_logits), B, V, V, B * V, bufs["len"], B, T, w.h, bufs["ud"], bufs["act"],
                          bufs["tok"], bufs["ent"], bufs["stop"], bufs["stats"], stream=body)
        if apart:
            ctx.pack_ragged(bufs["len"], B, K_cap, bufs["cu"], stream=body)
        ctx.policy_advance(policy, bufs["stop"], bufs["gamma"], bufs["len"], bufs["act"], B, K_cap, bufs["nact"], stream=body)
        ctx.graph_loop_end()
        graph = ctx.graph_end(st)
        assert ctx.launch_count() - before == (3 if apart else 1)    # draft step, packing, policy step, or the draft step alone
        seen = []
        for replay in range(2):                                      # the second one starts where the first one ended
            graph.launch(st)
            st.synchronize()
            seen.append([bufs[k].cpu().numpy().copy() for k in ("len", "act", "nact", "tok", "ent", "stop", "stats")])
            bufs["act"].fill_(1); bufs["len"].fill_(0)
            torch.cuda.synchronize()
        graph.destroy()
        got.append(seen)
    ctx.read_status()          # packing a length of 0 sets a bit
    for a, b in zip(*got):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
