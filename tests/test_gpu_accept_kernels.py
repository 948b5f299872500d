"""Acceptance where a slice's exponentials have no room on chip, and the kernels for one and for two blocks per SM against each
other.

A tree's acceptance lengths come from the kernel for one block per SM when it is alone and from the one for two when it is one of
many; both deal its rows out to the same number of blocks.  The walk's blocks per sequence depend on the batch, so there the
sums' order differs and only what is decided is compared."""
import pytest

from paper_2512_14069_b200 import binding as rb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return rb.Context(0)


def _tree(torch, V, dtype, seed):
    """One tree of 21 rows, five with children (of one child to eight), and its logits, among them zeros of both signs, numbers
    below fp32's normal range and -inf."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    parent = [-1] + [0] * 5 + [1] * 8 + [2] * 4 + [6] + [18] * 2
    depth = [0]
    for p in parent[1:]:
        depth.append(depth[p] + 1)
    tok = torch.randperm(V, device="cuda", generator=g)[:21].int()
    draft_row = [min(i, 7) for i in range(21)]
    z = torch.randn(2, 64, V, device="cuda", generator=g) * 2
    z[:, :, 3::7] = 0.0
    z[:, :, 5::11] = -0.0
    z[:, :, 6::13] = 1e-41
    z[:, :, 8::17] = -float("inf")
    z[0, 1, : V // 2] -= 300.0                       # a row with a wide range
    return z[0].to(dtype), z[1, :8].to(dtype), tok, parent, depth, draft_row


def _batch(torch, B, trees):
    pad = lambda x, v: torch.tensor([list(x) + [v] * (64 - len(x))], dtype=torch.int32, device="cuda")
    rows = [trees[b % len(trees)] for b in range(B)]
    return dict(target_logits=torch.stack([t[0] for t in rows]).contiguous(), draft_logits=torch.stack([t[1] for t in rows]).contiguous(),
                tree_tok=torch.cat([pad(t[2].tolist(), -1) for t in rows]), tree_parent=torch.cat([pad(t[3], -1) for t in rows]),
                tree_draft_row=torch.cat([pad(t[5], -1) for t in rows]), n_nodes=torch.full((B,), 21, dtype=torch.int32, device="cuda")), \
        torch.cat([pad(t[4], 0) for t in rows])


def _lengths(torch, ctx, B, V, T, trees):
    args, depth = _batch(torch, B, trees)
    dist = torch.empty(B, 6, dtype=torch.float64, device="cuda")
    acc = torch.empty(B, 64, dtype=torch.float64, device="cuda")
    ws = torch.full((rb.radar_acclen_workspace_bytes(ctx, B, V) + 256,), 0xff, dtype=torch.uint8, device="cuda")
    ws = ws[-ws.data_ptr() % 256:][:rb.radar_acclen_workspace_bytes(ctx, B, V)]
    rb.radar_accept_length_distribution(ctx, B=B, V=V, t_max=5, temperature=T, R=8, tree_depth=depth, dist=dist, p_acc_node=acc, workspace=ws, **args)
    return dist, acc, ctx.read_device_status()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,T", [(257, 1.0), (5003, 0.03), (5003, 1e-3), (5003, 2.0 ** -127), (5003, 2.0 ** -130), (5003, 3e38), (54016, 1.0), (70001, 0.7), (128256, 1.0)])
def test_acceptance_lengths_of_one_tree_and_of_many(ctx, dtype, V, T):
    import torch
    trees = [_tree(torch, V, torch.float32 if dtype == "f32" else torch.bfloat16, V + i) for i in range(2)]
    many, acc, status = _lengths(torch, ctx, 18, V, T, trees)
    assert status == 0 and bool(torch.isfinite(many).all())
    for i in range(2):
        one, acc1, status = _lengths(torch, ctx, 1, V, T, trees[i:i + 1])
        assert status == 0
        assert abs(float(one.sum()) - 1.0) < 1e-9
        # same exponentials, same order of sums: rounding of the scalars' products at most
        assert float((many[i::2] - one).abs().max()) < 1e-12 and float((acc[i::2] - acc1).abs().max()) < 1e-12


def test_acceptance_lengths_against_probabilities(ctx):
    """The root's first child is accepted with min(1, p / q); the spilled slice's sums are those of fp64 softmax."""
    import torch
    V = 128256
    for dtype, B in ((torch.float32, 1), (torch.float32, 9), (torch.bfloat16, 9)):
        t = _tree(torch, V, dtype, 7)
        p, q = torch.softmax(t[0][0].double(), -1), torch.softmax(t[1][0].double(), -1)
        x = int(t[2][1])
        _, acc, status = _lengths(torch, ctx, B, V, 1.0, [t])
        assert status == 0
        assert float((acc[:, 1] - min(1.0, float(p[x] / q[x]))).abs().max()) < 1e-9


@pytest.mark.parametrize("B", [1, 18])
def test_acceptance_lengths_report_nan(ctx, B):
    import torch
    for at in (0, 6000, 11001):
        t = _tree(torch, 11003, torch.float32, 3)
        t[0][2, at] = float("nan")
        assert _lengths(torch, ctx, B, 11003, 1.0, [t])[2] == -6
        assert ctx.read_device_status() == 0


def _walk(torch, ctx, B, V, T, trees, u):
    args, _ = _batch(torch, B, trees)
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
    out = dict(accept_len=i32(B), path_nodes=i32(B, 6), path_tokens=i32(B, 6), next_token=i32(B), best_retrieve_row=i32(B))
    need = rb.radar_accept_workspace_bytes(ctx, B, V, rb.RADAR_STOCHASTIC)
    ws = torch.full((need + 256,), 0xff, dtype=torch.uint8, device="cuda")
    ws = ws[-ws.data_ptr() % 256:][:need]
    retrieve = torch.full((B, 8, 6), -1, dtype=torch.int32, device="cuda")
    rb.radar_verify_accept(ctx, B=B, V=V, N=8, t_max=5, R=8, mode=rb.RADAR_STOCHASTIC, temperature=T, retrieve=retrieve,
                           n_leaves=torch.full((B,), 8, dtype=torch.int32, device="cuda"), u_accept=u[0][torch.arange(B) % len(trees)].contiguous(),
                           u_sample=u[1][torch.arange(B) % len(trees)].contiguous(), workspace=ws, **args, **out)
    return out, ctx.read_device_status()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,T", [(5003, 0.5), (54016, 1.0), (70001, 0.7), (128256, 1.0)])
def test_walks_of_one_sequence_and_of_many(ctx, dtype, V, T):
    import torch
    n = 4
    trees = [_tree(torch, V, torch.float32 if dtype == "f32" else torch.bfloat16, 2 * V + i) for i in range(n)]
    g = torch.Generator(device="cuda").manual_seed(V)
    u = torch.rand(n, 64, device="cuda", generator=g), torch.rand(n, device="cuda", generator=g)
    many, status = _walk(torch, ctx, 32, V, T, trees, u)
    assert status == 0
    for i in range(n):
        one, status = _walk(torch, ctx, 1, V, T, trees[i:i + 1], (u[0][i:i + 1], u[1][i:i + 1]))
        assert status == 0
        for k in one:
            assert torch.equal(many[k][i::n], one[k].expand_as(many[k][i::n])), k
