"""The draft calls of a step in ranges (radar_expand_range) against the same calls one by one (radar_expand_step): every cut of a
step into ranges, sequences that stop at, before and behind a range's ends, the three policies, most scores, NaN rows, a pool
that ends inside a range; and the rows' top-k where their bound changes.

Whole numbers must agree.  Both forms run the same passes and merges, so floats differ by the order of the gate's input-side
sums at most: 1e-6 on scores in [0, 1] and logits of order 1."""
import numpy as np
import pytest

from paper_2512_14069_b200 import workloads as W
from test_gpu_expand_calls import NAMES, ctx       # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def _run(ctx, draft, k, t_max, ranges, policy, force, features=None, capacity=None):     # noqa: F811
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    B, _, V = draft.shape
    cfg = W.shrink(W.CONFIGS[2], k=k, t_max=t_max)
    w = W.gate_weights(cfg) if policy == 0 else W.policy_weights(cfg, ("mlp_scores", "lstm_hidden")[policy - 1], 64)
    gate = {n: torch.from_numpy(x).cuda() for n, x in w.items()}
    s = SpecStep(ctx, B=B, V=V, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16, logits_dtype=draft.dtype)
    s.C = capacity or s.C
    for _ in range(2):                               # the second step finds the first one's state and workspace
        if ranges:
            s.ranges = ranges
            s.ws_calls = torch.full((max(rb.radar_expand_range_workspace_bytes(ctx, B, V, k, *r) for r in ranges),), 0xff, dtype=torch.uint8, device="cuda")
        s.run_expansion(draft, gate, force, policy, features, pipelined=bool(ranges))
    status = ctx.read_device_status()
    return s, status


def _same(a, b):
    for n in NAMES:
        x, y = getattr(a, n).cpu(), getattr(b, n).cpu()
        if x.dtype.is_floating_point:
            np.testing.assert_allclose(y.numpy(), x.numpy(), rtol=0, atol=1e-6, err_msg=n)
        else:
            assert np.array_equal(x.numpy(), y.numpy()), n


@pytest.mark.parametrize("policy", [0, 1, 2])
@pytest.mark.parametrize("t_max,ranges", [(1, [(1, 1)]), (2, [(1, 1), (2, 2)]), (3, [(1, 2), (3, 3)]), (6, [(1, 6)]), (6, [(1, 1), (2, 6)]),
                                          (6, [(1, 2), (3, 5), (6, 6)]), (6, [(1, 3), (4, 6)]), (6, [(1, 5), (6, 6)]), (6, [(t, t) for t in range(1, 7)])])
def test_ranges_match_one_by_one(ctx, policy, t_max, ranges):     # noqa: F811
    import torch
    B, V, k = 9, 3000, 5
    g = torch.Generator(device="cuda").manual_seed(t_max * 10 + policy)
    draft = torch.randn(B, 1 + (t_max - 1) * k, V, device="cuda", generator=g) * 3
    features = torch.randn(max(t_max - 1, 1), B, 64, device="cuda", generator=g) if policy == 2 else None
    for force in (torch.arange(B, dtype=torch.int32, device="cuda") % t_max + 1, None):
        one, _ = _run(ctx, draft, k, t_max, None, policy, force, features)
        some, status = _run(ctx, draft, k, t_max, ranges, policy, force, features)
        assert status == 0
        _same(one, some)


@pytest.mark.parametrize("k", [1, 32])
def test_fewest_and_most_scores(ctx, k):     # noqa: F811
    import torch
    draft = torch.randn(3, 1 + 4 * k, 2000, device="cuda").to(torch.bfloat16)          # (many equal values)
    force = torch.tensor([5, 2, 3], dtype=torch.int32, device="cuda")
    one, _ = _run(ctx, draft, k, 5, None, 0, force)
    some, status = _run(ctx, draft, k, 5, [(1, 2), (3, 5)], 0, force)
    assert status == 0
    _same(one, some)


def test_nan_rows_and_a_small_pool(ctx):     # noqa: F811
    import torch
    k, t_max = 4, 5
    draft = torch.randn(2, 1 + (t_max - 1) * k, 1000, device="cuda")
    force = torch.full((2,), t_max, dtype=torch.int32, device="cuda")
    s, status = _run(ctx, draft, k, t_max, [(1, 2), (3, 5)], 0, force, capacity=k + 2 * k * k)      # room for three calls
    assert status == -1 and s.pool_len.cpu().tolist() == [k + 2 * k * k] * 2
    assert s.cont_hist.cpu().numpy().tolist() == [[1, 1], [1, 1], [1, 1], [0, 0], [0, 0]] and s.active.cpu().tolist() == [0, 0]
    draft[1, 1 + 3 * k:] = float("nan")              # rows of call 5, which sequence 1 does not make
    assert _run(ctx, draft, k, t_max, [(1, 2), (3, 5)], 0, torch.tensor([5, 4], dtype=torch.int32, device="cuda"))[1] == 0
    assert _run(ctx, draft, k, t_max, [(1, 2), (3, 5)], 0, force)[1] == -6


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [32, 263, 1024, 1028, 8191, 8200, 40000, 170001])
@pytest.mark.parametrize("k", [1, 10, 32])
def test_rows_top_k(ctx, dtype, V, k):     # noqa: F811
    """Rows with few finite values (fewer than k; all in one span; one in every span), with ties beyond the lists' room, and
    rows that start off a 16-byte boundary."""
    import torch
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = torch.randn(7, V, device="cuda", generator=g)
    x[1, :] = float("-inf"); x[1, V // 2::max(V // 4, 1)] = 1.0
    x[2, :] = float("-inf"); x[2, V - min(V, 200):] = torch.randn(min(V, 200), device="cuda", generator=g)
    x[3, :] = float("-inf"); x[3, 5::1024] = torch.randn(len(x[3, 5::1024]), device="cuda", generator=g)
    x[4, :] = 0.5
    x[5, ::3] = 7.0
    draft = x.to(dt).view(7, 1, V)
    s, status = _run(ctx, draft, k, 1, [(1, 1)], 0, None)
    assert status == 0
    ref = draft[:, 0].double()
    order = torch.sort(ref, dim=-1, descending=True, stable=True).indices[:, :k]
    assert torch.equal(s.topk_tok1[:, 0].long(), order)
    lp = torch.log_softmax(ref, -1).gather(1, order)
    got = s.topk_logp1[:, 0].double()
    assert torch.equal(got == float("-inf"), lp == float("-inf"))
    fin = torch.isfinite(lp)
    assert float((got - lp)[fin].abs().max()) < 2e-6 + 16 * 2 ** -24


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,k", [(32, 32), (263, 10), (1028, 1), (8200, 10), (40000, 32), (131073, 4), (170001, 10), (270001, 32)])
def test_many_rows_top_k(ctx, dtype, V, k):     # noqa: F811
    """The same kinds of rows where there are too many of them for a cluster each (301 > 2 * 148): pass and merge kernels,
    longer rows than 128 spans, and every row of an odd V at another distance from a 16-byte boundary."""
    import torch
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = torch.randn(7, V, device="cuda", generator=g)
    x[1, :] = float("-inf"); x[1, V // 2::max(V // 4, 1)] = 1.0
    x[2, :] = float("-inf"); x[2, V - min(V, 200):] = torch.randn(min(V, 200), device="cuda", generator=g)
    x[3, :] = float("-inf"); x[3, 5::1024] = torch.randn(len(x[3, 5::1024]), device="cuda", generator=g)
    x[4, :] = 0.5
    x[5, ::3] = 7.0
    x = x.to(dt)
    s, status = _run(ctx, x.repeat(43, 1).view(301, 1, V), k, 1, None, 0, None)
    assert status == 0
    order = torch.sort(x.double(), dim=-1, descending=True, stable=True).indices[:, :k]
    assert torch.equal(s.topk_tok1[:, 0].long().view(43, 7, k), order.expand(43, 7, k))
    lp = torch.log_softmax(x.double(), -1).gather(1, order).expand(43, 7, k)
    got = s.topk_logp1[:, 0].double().view(43, 7, k)
    assert torch.equal(got == float("-inf"), lp == float("-inf"))
    fin = torch.isfinite(lp)
    assert float((got - lp)[fin].abs().max()) < 2e-6 + 16 * 2 ** -24
