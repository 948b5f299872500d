"""radar_expand_step with a pool that has no room for a sequence's candidates: the call reports it and leaves pool and frontier
alone, and the rows' top-k, which needs no pool, is there for every sequence; a NaN row is still reported before it.  One block
a sequence and the cluster with helper blocks."""
import pytest

from paper_2512_14069_b200 import workloads as W
from test_gpu_expand_calls import ctx       # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,V,k,policy", [(2, 3000, 5, 0), (2, 3000, 5, 1), (5, 128256, 8, 0)])
@pytest.mark.parametrize("nan", [False, True])
def test_top_k_of_a_sequence_without_room(ctx, B, V, k, policy, nan):     # noqa: F811
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    t_max = 3
    g = torch.Generator(device="cuda").manual_seed(V)
    draft = torch.randn(B, 1 + (t_max - 1) * k, V, device="cuda", generator=g) * 3
    cfg = W.shrink(W.CONFIGS[2], k=k, t_max=t_max)
    w = W.gate_weights(cfg) if policy == 0 else W.policy_weights(cfg, "mlp_scores")
    gate = {n: torch.from_numpy(x).cuda() for n, x in w.items()}
    force = torch.full((B,), t_max, dtype=torch.int32, device="cuda")
    s = SpecStep(ctx, B=B, V=V, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
    s.expand(1, draft, gate, force, policy)
    ctx.check_device_status()
    s.pool_len[1] = s.C - k * k + 1                  # sequence 1: one entry too few
    before = {n: getattr(s, n)[1].clone() for n in ("pool_tok", "pool_score", "pool_draft_row")}
    if nan:
        draft[1, 1 + k - 1, 17] = float("nan")
    s.expand(2, draft, gate, force, policy)
    assert ctx.read_device_status() == (-6 if nan else -1)
    rows = draft[:, 1:1 + k].double()
    order = torch.sort(rows, dim=-1, descending=True, stable=True).indices[..., :k]
    good = torch.ones(B, k, dtype=torch.bool, device="cuda")
    good[1, k - 1] = not nan                         # (what a NaN row gives is not specified)
    assert torch.equal(s.topk_tok[1].long()[good], order[good])
    lp = torch.log_softmax(rows, -1).gather(-1, order)
    assert float((s.topk_logp[1].double() - lp)[good].abs().max()) < 2e-6 + 16 * 2 ** -24
    for n, x in before.items():
        assert torch.equal(getattr(s, n)[1], x), n
    assert int(s.pool_len[1]) == s.C - k * k + 1 and not int(s.active[1]) and not int(s.cont_hist[1, 1])
    assert bool((s.frontier_tok[1, 1] == 0).all()) and int(s.active[0]) == 1
