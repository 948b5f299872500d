"""Launches whose static and dynamic shared memory together pass 48 KB while the dynamic part alone does not, each on a new
context, and two contexts of one device that take turns with large and small launches of one kernel."""
import numpy as np
import pytest

import harness as H
from paper_2512_14069_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [11, 12, 14, 16, 23, 24, 32])
@pytest.mark.parametrize("t_max,policy", [(1, 0), (1, 1), (3, 0), (3, 1)])
def test_expansion_on_a_new_context(k, t_max, policy):
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    cfg = W.shrink(W.CONFIGS[2], k=k, t_max=t_max)
    gate = {n: H.to_dev(x) for n, x in (W.policy_weights(cfg, "mlp_scores") if policy else W.gate_weights(cfg)).items()}
    draft = torch.randn(2, 1 + (t_max - 1) * k, 3000, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k)) * 3
    got = []
    for pipelined in (True, False):
        ctx = rb.Context(0)
        s = SpecStep(ctx, B=2, V=3000, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
        s.run_expansion(draft, gate, torch.full((2,), t_max, dtype=torch.int32, device="cuda"), policy, pipelined=pipelined)
        ctx.check_device_status()
        got.append([x.cpu().numpy() for x in (s.pool_tok, s.pool_parent, s.frontier_tok, s.pool_len)])
        ctx.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("C", [2047, 2472, 2560, 2688, 2700, 8192])
def test_tree_of_a_pool_on_a_new_context(C):
    """Pools of one call's candidates (all children of the root), fewer of them live than fit: the N best, in pool order."""
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx = rb.Context(0)
    i32 = dict(dtype=torch.int32, device="cuda")
    score = torch.randn(1, C, device="cuda", generator=torch.Generator(device="cuda").manual_seed(C))
    N, L = 63, C - 3
    out = {n: torch.zeros(1, 64, **i32) for n in ("tree_tok", "tree_parent", "tree_depth", "tree_pos", "tree_pool_idx", "tree_draft_row")}
    n_nodes = torch.zeros(1, **i32)
    rb.radar_rerank_build_tree(
        ctx, B=1, N=N, t_max=4, pool_capacity=C, pool_tok=torch.arange(C, **i32)[None], pool_parent=torch.full((1, C), -1, **i32),
        pool_depth=torch.ones(1, C, **i32), pool_draft_row=torch.full((1, C), -1, **i32), pool_score=score,
        pool_len=torch.tensor([L], **i32), root_tok=torch.zeros(1, **i32), prefix_len=torch.zeros(1, **i32),
        tree_score=torch.zeros(1, 64, device="cuda"), tree_mask=torch.zeros(1, 64, dtype=torch.int64, device="cuda"), n_nodes=n_nodes,
        retrieve=torch.zeros(1, N, 5, **i32), n_leaves=torch.zeros(1, **i32), **out)
    ctx.check_device_status()
    want = sorted(np.argsort(-score[0, :L].cpu().numpy(), kind="stable")[:N].tolist())
    assert int(n_nodes) == N + 1 and out["tree_pool_idx"].cpu().tolist()[0][1:] == want
    ctx.close()


def test_two_contexts_take_turns():
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep

    def step(ctx, k):
        cfg = W.shrink(W.CONFIGS[2], k=k, t_max=2)
        gate = {n: H.to_dev(x) for n, x in W.gate_weights(cfg).items()}
        s = SpecStep(ctx, B=1, V=20000, k=k, t_max=2, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
        draft = torch.randn(1, s.R, 20000, device="cuda")
        return lambda: s.run_expansion(draft, gate, pipelined=False)
    one, two = rb.Context(0), rb.Context(0)
    large, small = step(one, 32), step(two, 2)
    for run in (large, small, large):                # the second context's first launch is smaller than the first one's
        run()
    one.check_device_status()
    two.check_device_status()
    one.close()
    two.close()
