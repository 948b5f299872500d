"""All draft calls of a step in one go (radar_expand_calls) against the same calls one by one (radar_expand_step): fewest and
most calls and scores, sequences that stop at every call, forced and by the gate, both score policies, ties that make every
candidate a survivor, NaN rows of calls that are and are not made, a pool that is too small, and the line above which the
calls go one by one.

Whole numbers must agree.  The two forms may cut a row into different chunks, whose fp32 sums of at most 8192
exponentials are each off by at most some 16 ulp: a log-probability by 2e-6, a cumulative score by that a call, and the gate
(weights of a few tenths, scores in [0, 1]) by a small multiple of it."""
import numpy as np
import pytest

from paper_2512_14069_b200 import workloads as W

pytestmark = pytest.mark.gpu
NAMES = ("pool_tok", "pool_parent", "pool_depth", "pool_draft_row", "pool_score", "pool_len", "frontier_tok", "frontier_score",
         "frontier_pool_idx", "frontier_src_row", "topk_tok", "topk_logp", "topk_tok1", "topk_logp1", "gate_logits", "cont_hist", "h", "c",
         "active")


@pytest.fixture(scope="module")
def ctx():
    from paper_2512_14069_b200 import binding as rb
    c = rb.Context(0)
    yield c
    c.close()


def _step(ctx, B, V, k, t_max):
    import torch
    from paper_2512_14069_b200.pipeline import SpecStep
    return SpecStep(ctx, B=B, V=V, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)


def _gate(k, t_max, policy):
    import torch
    cfg = W.shrink(W.CONFIGS[2], k=k, t_max=t_max)
    w = W.policy_weights(cfg, "mlp_scores") if policy == 1 else W.gate_weights(cfg)
    return {n: torch.from_numpy(x).cuda() for n, x in w.items()}


def _both(ctx, draft, k, t_max, gate, force, policy, check=True):
    B, _, V = draft.shape
    one, all_ = _step(ctx, B, V, k, t_max), _step(ctx, B, V, k, t_max)
    assert all_.ws_calls is not None
    for _ in range(2):                                   # the second step finds the first one's state and workspace
        one.run_expansion(draft, gate, force, policy, pipelined=False)
        all_.run_expansion(draft, gate, force, policy)
        if check:
            ctx.check_device_status()
    for n in NAMES:
        x, y = getattr(one, n).cpu(), getattr(all_, n).cpu()
        if x.dtype.is_floating_point:
            np.testing.assert_allclose(y.numpy(), x.numpy(), rtol=0, atol=1e-5 * t_max, err_msg=n)
        else:
            assert np.array_equal(x.numpy(), y.numpy()), n
    return all_


@pytest.mark.parametrize("B,V,k,t_max,policy", [(1, 40, 1, 1, 0), (3, 5000, 4, 2, 0), (5, 9000, 10, 3, 0), (9, 9000, 10, 8, 0),
                                                (17, 2000, 7, 16, 0), (2, 9000, 12, 6, 0), (4, 3000, 16, 4, 0), (2, 33000, 32, 16, 0), (6, 9000, 10, 8, 1), (3, 3000, 1, 5, 0)])
def test_calls_together_match_one_by_one(ctx, B, V, k, t_max, policy):
    import torch
    g = torch.Generator(device="cuda").manual_seed(B * V + k)
    draft = torch.randn(B, 1 + (t_max - 1) * k, V, device="cuda", generator=g) * 3
    gate = _gate(k, t_max, policy)
    force = torch.arange(B, dtype=torch.int32, device="cuda") % t_max + 1          # a stop at every call
    s = _both(ctx, draft, k, t_max, gate, force, policy)
    assert s.pool_len.cpu().tolist() == [k + b % t_max * k * k for b in range(B)]
    _both(ctx, draft, k, t_max, gate, None, policy)                                # ... and where the gate stops


@pytest.mark.parametrize("k", [4, 32])
def test_ties_make_every_candidate_a_survivor(ctx, k):
    import torch
    draft = torch.zeros(2, 1 + 3 * k, 500, device="cuda")
    _both(ctx, draft, k, 4, _gate(k, 4, 0), torch.full((2,), 4, dtype=torch.int32, device="cuda"), 0)


def test_nan_rows_count_where_the_call_is_made(ctx):
    import torch
    from paper_2512_14069_b200 import binding as rb
    B, V, k, t_max = 3, 3000, 5, 6
    draft = torch.randn(B, 1 + (t_max - 1) * k, V, device="cuda")
    gate = _gate(k, t_max, 0)
    force = torch.tensor([2, 3, 6], dtype=torch.int32, device="cuda")
    draft[0, 1 + 1 * k:] = float("nan")                  # sequence 0 makes two calls: rows 0 .. k
    draft[1, 1 + 2 * k, 17] = float("nan")
    _both(ctx, draft, k, t_max, gate, force, 0)
    draft[1, 1 + 1 * k + 2, 2999] = float("nan")         # a row of sequence 1's third call
    s = _step(ctx, B, V, k, t_max)
    s.run_expansion(draft, gate, force)
    with pytest.raises(rb.RadarError) as err:
        ctx.check_device_status()
    assert err.value.status == -6


def test_pool_that_is_too_small_stops_the_sequence(ctx):
    import torch
    from paper_2512_14069_b200 import binding as rb
    B, V, k, t_max = 2, 1000, 4, 4
    s = _step(ctx, B, V, k, t_max)
    s.C = k + k * k                                      # room for two calls (the buffers hold four)
    s.run_expansion(torch.randn(B, s.R, V, device="cuda"), _gate(k, t_max, 0), torch.full((B,), 4, dtype=torch.int32, device="cuda"))
    with pytest.raises(rb.RadarError) as err:
        ctx.check_device_status()
    assert err.value.status == -1
    assert s.pool_len.cpu().tolist() == [s.C] * B and s.active.cpu().tolist() == [0] * B
    assert s.cont_hist.cpu().numpy().tolist() == [[1, 1], [1, 1], [0, 0], [0, 0]]


def test_long_passes_go_call_by_call(ctx):
    from paper_2512_14069_b200 import binding as rb
    assert rb.radar_expand_calls_workspace_bytes(ctx, 1, 128256, 10, 8) > 0
    assert rb.radar_expand_calls_workspace_bytes(ctx, 32, 128256, 10, 8) == 0
    assert rb.radar_expand_calls_workspace_bytes(ctx, 1, 1 << 19, 8, 2) > 0 and rb.radar_expand_calls_workspace_bytes(ctx, 1, (1 << 19) + 1, 8, 2) == 0
    assert rb.radar_expand_calls_workspace_bytes(ctx, 1, 1000, 33, 8) == 0


def test_a_workspace_full_of_other_sizes(ctx):
    """Nothing of the workspace is read before it has been written: one that other sizes, and NaN patterns, have left behind."""
    import torch
    V, k, t_max = 9000, 10, 5
    big = _step(ctx, 6, 30000, 12, 6)
    big.run_expansion(torch.randn(6, big.R, 30000, device="cuda"), _gate(12, 6, 0))
    draft = torch.randn(3, 1 + (t_max - 1) * k, V, device="cuda") * 3
    gate, got = _gate(k, t_max, 0), []
    for fill in (None, 0xff, 0):
        s = _step(ctx, 3, V, k, t_max)
        if fill is None:
            s.ws_calls = big.ws_calls
        else:
            s.ws_calls.fill_(fill)
        s.run_expansion(draft, gate)
        ctx.check_device_status()
        got.append([getattr(s, n).cpu() for n in NAMES])
    for other in got[:2]:
        assert all(torch.equal(x, y) for x, y in zip(got[2], other))
