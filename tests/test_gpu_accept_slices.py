"""Stochastic acceptance and Eq. 11-13 where a sequence's (a tree row's) vocabulary is cut into the slices of a cluster:
vocabularies around a quad, around the sizes at which the cluster grows, unaligned rows, and logits spread over more
than the range of fp64 exponentials.  Decisions exact against the oracle; distributions within 1e-11 (both sides sum V
fp64 terms in their own order: V 2^-53 = 7e-12 at V = 65540)."""
import numpy as np
import pytest

import harness as H
from paper_2512_14069_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2512_14069_b200 import binding as rb
    c = rb.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("V,k,spread,bf16", [
    (5, 2, 1.0, False), (7, 4, 1.0, False), (1000, 4, 500.0, False), (2050, 4, 1.0, True), (4096, 4, 1.0, False),
    (8195, 8, 1.0, True), (16387, 8, 1.0, False), (32770, 8, 700.0, False), (65540, 4, 1.0, False)])
def test_slices(ctx, V, k, spread, bf16):
    import torch
    from oracle import accept_oracle as A
    from paper_2512_14069_b200 import binding as rb
    cfg = W.shrink(W.CONFIGS[3], cid=500 + V % 97, B=3, V=V, k=k, t_max=4, N=min(24, k + 3 * k * k), depth_plan="fixed_tmax", temperature=0.7)
    inp = H.make_inputs(cfg, with_attention=False)
    rnd = (lambda x: W.bf16_bits_to_f32(W.f32_to_bf16_bits(x)).reshape(x.shape)) if bf16 else (lambda x: x)
    inp["draft"] = rnd(inp["draft"])
    pools, traces, trees = H.oracle_expand_and_tree(cfg, inp)
    target = H.make_target(cfg, inp, trees)
    # every third token far below the rest: exponentials near and past the smallest fp64 numbers
    far = np.arange(V) % 3 == 2
    low = np.where(far, np.float32(spread - 1.0), np.float32(0.0)).astype(np.float32)
    target, draft = rnd(target - low), rnd(inp["draft"] - low)
    inp["draft"] = draft
    accepts = H.oracle_accept(cfg, inp, trees, target)
    g = H.CudaRun(cfg, dict(inp), ctx, logits_bf16=bf16)
    s = g.step
    # the oracle's trees, whatever the draft logits have become
    pad = lambda x, fill: np.pad(np.asarray(x[:64]), (0, max(0, 64 - len(x))), constant_values=fill).astype(np.int32)
    for name, key, fill in (("tree_tok", "tok", -1), ("tree_parent", "parent", -1), ("tree_depth", "depth", 0), ("tree_draft_row", "draft_row", -1)):
        getattr(s, name).copy_(H.to_dev(np.stack([pad(t[key], fill) for t in trees])))
    s.n_nodes.copy_(H.to_dev(np.array([t["n_nodes"] for t in trees], np.int32)))
    s.n_leaves.copy_(H.to_dev(np.array([t["n_leaves"] for t in trees], np.int32)))
    s.retrieve.copy_(H.to_dev(np.stack([np.asarray(t["retrieve"]) for t in trees]).astype(np.int32)))
    for a in accepts:                                  # no decision of the oracle within rounding of a tie
        assert a["accept_margin"] > H.TAU_PROB and a["sample_margin"] > H.TAU_PROB
    g.accept(target)
    H.compare_accept(cfg, g, accepts)

    T = float(np.float32(cfg.temperature))
    dist = torch.full((cfg.B, cfg.t_max + 1), -1.0, dtype=torch.float64, device="cuda")
    pacc = torch.full((cfg.B, 64), -1.0, dtype=torch.float64, device="cuda")
    ws = torch.zeros(rb.radar_acclen_workspace_bytes(ctx, cfg.B, V), dtype=torch.uint8, device="cuda")
    tl = H.to_dev(target)
    rb.radar_accept_length_distribution(
        ctx, B=cfg.B, V=V, t_max=cfg.t_max, temperature=T, target_logits=tl.to(torch.bfloat16) if bf16 else tl, tree_tok=s.tree_tok,
        tree_parent=s.tree_parent, tree_depth=s.tree_depth, tree_draft_row=s.tree_draft_row, n_nodes=s.n_nodes, draft_logits=g.draft,
        R=s.R, dist=dist, p_acc_node=pacc, workspace=ws)
    ctx.check_device_status()
    dist, pacc = dist.cpu().numpy(), pacc.cpu().numpy()
    for b in range(cfg.B):
        d_ref, p_ref = A.accept_length_distribution(target[b], draft[b], trees[b], T, cfg.t_max)
        n = trees[b]["n_nodes"]
        assert np.max(np.abs(dist[b] - d_ref)) < 1e-11 and np.max(np.abs(pacc[b, :n] - p_ref)) < 1e-11 and not pacc[b, n:].any()
