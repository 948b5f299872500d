"""Rerank and serialisation over pools at the edges of the selection: fewer entries than nodes, fewer than a warp, one past a
warp, up to and just past the 1024 entries the one-entry-a-thread form takes, distinct scores and scores with many ties.
All outputs are whole numbers or copies, compared exactly with a plain restatement in numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
T_MAX = 8


def _pool(rng, L, ties):
    parent, depth = np.full(L, -1, np.int32), np.ones(L, np.int32)
    score = np.zeros(L, np.float32)
    for i in range(L):
        p = -1 if i < 3 else int(rng.integers(-1, i))
        while p >= 0 and depth[p] >= T_MAX:
            p = int(parent[p])
        parent[i], depth[i] = p, 1 if p < 0 else depth[p] + 1
        step = np.float32(rng.integers(0, 3)) if ties else np.float32(rng.exponential())
        score[i] = (0 if p < 0 else score[p]) - step
    return parent, depth, score


def _reference(parent, depth, score, tok, drow, n, root, plen, N, W):
    order = sorted(range(len(score)), key=lambda i: (-score[i], i))[:n]
    kept = sorted(order)
    row = {i: r + 1 for r, i in enumerate(kept)}
    M = len(kept) + 1
    par = [-1] + [row[parent[i]] if parent[i] >= 0 else 0 for i in kept]
    dep = [0] + [int(depth[i]) for i in kept]
    has = [r in par for r in range(M)]
    paths = []
    for r in range(M):
        p, j = [], r
        while j >= 0:
            p.append(j)
            j = par[j]
        paths.append(p[::-1])
    leaves = [r for r in range(M) if not has[r]] if M > 1 else []
    dr = [0] + [int(drow[i]) for i in kept]
    ret = np.full((N, W), -1)
    for l, r in enumerate(leaves):
        ret[l, :len(paths[r])] = paths[r]
    return dict(tree_tok=[root] + [int(tok[i]) for i in kept], tree_parent=par, tree_depth=dep, tree_pos=[plen + d for d in dep],
                tree_pool_idx=[-1] + kept, tree_score=[np.float32(0)] + [score[i] for i in kept],
                tree_draft_row=[dr[r] if has[r] else -1 for r in range(M)],
                tree_mask=[sum(1 << j for j in paths[r]) for r in range(M)]), M, leaves, ret


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("N", [1, 32, 33, 63])
def test_pool_sizes(N, ties):
    import torch
    from paper_2512_14069_b200 import binding as rb
    rng = np.random.default_rng(N + 100 * ties)
    sizes = [0, 1, 5, 31, 32, 33, 62, 63, 64, 65, 500, 1023, 1024, 1025, 2000]
    B, C, W = len(sizes), 2000, T_MAX + 1
    parent, depth, score = np.full((B, C), 7, np.int32), np.full((B, C), 9, np.int32), np.full((B, C), 5, np.float32)   # stale past L
    for b, L in enumerate(sizes):
        parent[b, :L], depth[b, :L], score[b, :L] = _pool(rng, L, ties)
    tok, drow = rng.integers(0, 9999, (B, C)).astype(np.int32), rng.integers(-1, 70, (B, C)).astype(np.int32)
    root, plen = np.arange(B, dtype=np.int32) + 5, np.arange(B, dtype=np.int32) * 11
    keep = rng.integers(max(1, N // 2), N + 1, B).astype(np.int32)
    dev = lambda x: torch.from_numpy(x).cuda()
    z = lambda shape, dt=torch.int32: torch.full(shape, 3, dtype=dt, device="cuda")
    out = dict(tree_tok=z((B, 64)), tree_parent=z((B, 64)), tree_depth=z((B, 64)), tree_pos=z((B, 64)), tree_pool_idx=z((B, 64)),
               tree_draft_row=z((B, 64)), tree_score=z((B, 64), torch.float32), tree_mask=z((B, 64), torch.int64), n_nodes=z((B,)),
               retrieve=z((B, N, W)), n_leaves=z((B,)))
    ctx = rb.Context(0)
    rb.radar_rerank_build_tree(ctx, B=B, N=N, t_max=T_MAX, pool_capacity=C, pool_tok=dev(tok), pool_parent=dev(parent),
                               pool_depth=dev(depth), pool_draft_row=dev(drow), pool_score=dev(score),
                               pool_len=dev(np.asarray(sizes, np.int32)), n_keep=dev(keep), root_tok=dev(root), prefix_len=dev(plen), **out)
    ctx.check_device_status()
    got = {n: t.cpu().numpy() for n, t in out.items()}
    for b, L in enumerate(sizes):
        ref, M, leaves, ret = _reference(parent[b, :L], depth[b, :L], score[b, :L], tok[b], drow[b], min(int(keep[b]), L), int(root[b]),
                                         int(plen[b]), N, W)
        assert got["n_nodes"][b] == M and got["n_leaves"][b] == len(leaves), L
        for n, v in ref.items():
            x = got[n][b].view(np.uint64) if n == "tree_mask" else got[n][b]
            assert np.array_equal(x[:M], np.asarray(v, x.dtype)), (L, n)
            assert np.all(x[M:] == {"tree_depth": 0, "tree_pos": 0, "tree_score": 0, "tree_mask": 0}.get(n, np.asarray(-1).astype(x.dtype))), (L, n)
        assert np.array_equal(got["retrieve"][b], ret), L
    ctx.close()
