"""Stochastic acceptance and Eq. 11-13 over the range of temperatures: so near zero that neighbouring logits lie hundreds of units
of z / T apart (the exponentials' range test must not round such a logit into its range), and so large that z / T vanishes
(masked logits and the padding behind the vocabulary still weigh nothing).  Reference: fp64 softmax of (z - max) / T, the
difference of two logits being exact.  1e-11 as in the slices' test: |x| 2^-53 with |x| < 745 in the argument, 1.1 ulp of the
exponential, sums of at most 1003 terms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOK = (-1, 10, 500, 1002, 7, 998)
PARENT = (-1, 0, 0, 0, 1, 1)
DEPTH = (0, 1, 1, 1, 2, 2)
DRAFT_ROW = (0, 1, -1, -1, -1, -1)


def _softmax(z, T):
    z = z.astype(np.float64)
    e = np.exp((z - z.max()) / T)
    return e / e.sum()


def _children(target, draft, c, T):
    """[(row, P_acc(row | parent c), P(row proposed and accepted))] and the walk's weights behind every rejection."""
    p, q, reach, out = _softmax(target[c], T), _softmax(draft[DRAFT_ROW[c]], T), 1.0, []
    for j in [j for j in range(1, 6) if PARENT[j] == c]:
        x = TOK[j]
        acc = min(1.0, p[x] / q[x]) if q[x] > 0 else float(p[x] > 0)
        out.append((j, acc, reach * acc))
        reach *= 1.0 - acc
        r = np.maximum(0.0, p - q)
        p = r / r.sum() if r.sum() > 0 else p
        q = np.where(np.arange(q.size) == x, 0.0, q)
        if q.sum() <= 0:
            out += [(i, 0.0, 0.0) for i in range(j + 1, 6) if PARENT[i] == c]
            break
        q = q / q.sum()
    return out, p


@pytest.mark.parametrize("T,ref,steps,masked", [
    (1e-8, 20.0, 40, 0.0), (2e-8, 100.0, 40, 0.0), (2e-9, 2.5, 40, 0.0), (1e-8, -20.0, 40, 0.3), (1e-6, 20.0, 12, 0.0), (3e-7, 2.5, 9, 0.3),
    (1.0, 3.0, 0, 0.3), (4e35, 3.0, 0, 0.3), (1e36, 3.0, 0, 0.3), (3e38, 3.0, 0, 0.0)])
@pytest.mark.parametrize("V", [1003, 9001])
def test_temperature_range(T, ref, steps, masked, V):
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx, t_max, T = rb.Context(0), 3, float(np.float32(T))
    rng = np.random.default_rng(int(abs(ref) * 10) + steps + V)

    def rows(n):
        if steps:                                    # `steps` neighbouring values from ref downwards
            z = (np.float32(ref) - rng.integers(0, steps, (n, V)) * np.abs(np.spacing(np.float32(ref)))).astype(np.float32)
        else:
            z = rng.normal(ref, 1.0, (n, V)).astype(np.float32)
        z[rng.random((n, V)) < masked] = -np.inf
        return z
    target, draft = rows(64), rows(2)
    target[:, list(TOK[1:])], draft[:, list(TOK[1:])] = ref, ref              # the children are live tokens, with steps: of the best value
    dev = lambda x, dt=np.int32: torch.from_numpy(np.ascontiguousarray(np.asarray(x, dt))).cuda()
    pad = lambda x, fill: dev([list(x) + [fill] * (64 - len(x))])
    tok, par, dep, drow = pad(TOK, -1), pad(PARENT, -1), pad(DEPTH, 0), pad(DRAFT_ROW, -1)
    n_nodes, tl, dl = dev([6]), dev(target[None], np.float32), dev(draft[None], np.float32)

    dist, pacc = (torch.full((1, n), -1.0, dtype=torch.float64, device="cuda") for n in (t_max + 1, 64))
    ws = torch.zeros(rb.radar_acclen_workspace_bytes(ctx, 1, V), dtype=torch.uint8, device="cuda")
    rb.radar_accept_length_distribution(ctx, B=1, V=V, t_max=t_max, temperature=T, target_logits=tl, tree_tok=tok, tree_parent=par,
                                        tree_depth=dep, tree_draft_row=drow, n_nodes=n_nodes, draft_logits=dl, R=2, dist=dist,
                                        p_acc_node=pacc, workspace=ws)
    ctx.check_device_status()
    kids = {c: _children(target, draft, c, T) for c in (0, 1)}
    want = np.zeros(64)
    want[0] = 1.0
    for c in (0, 1):
        for j, _, p in kids[c][0]:
            want[j] = want[c] * p
    stop = want[:6] * (1.0 - np.array([sum(p for _, _, p in kids[c][0]) if c in kids else 0.0 for c in range(6)]))
    assert np.max(np.abs(pacc.cpu().numpy()[0] - want)) < 1e-11
    assert np.max(np.abs(dist.cpu().numpy()[0] - [sum(stop[i] for i in range(6) if DEPTH[i] == d) for d in range(t_max + 1)])) < 1e-11

    ws = torch.zeros(rb.radar_accept_workspace_bytes(ctx, 1, V, rb.RADAR_STOCHASTIC), dtype=torch.uint8, device="cuda")
    retrieve = np.full((1, 8, t_max + 1), -1)
    for l, r in enumerate([(0, 2), (0, 3), (0, 1, 4), (0, 1, 5)]):
        retrieve[0, l, :len(r)] = r
    retrieve, n_leaves = dev(retrieve), dev([4])
    alen, nxt, best = dev([0]), dev([0]), dev([0])
    nodes, toks = dev([[0] * (t_max + 1)]), dev([[0] * (t_max + 1)])
    for trial in range(6):
        u = rng.random(64).astype(np.float32)
        us = np.float32(rng.random())
        cur, path = 0, [0]
        while cur in kids:                           # the walk on the reference's probabilities
            took = None
            for j, acc, _ in kids[cur][0]:
                assert abs(float(u[j]) - acc) > 1e-9
                if u[j] < acc:
                    took = j
                    break
            if took is None:
                break
            cur = took
            path.append(cur)
        w = kids[cur][1] if cur in kids else _softmax(target[cur], T)
        cdf = np.cumsum(w)
        assert np.min(np.abs(cdf / cdf[-1] - float(us))) > 1e-9
        rb.radar_verify_accept(ctx, B=1, V=V, t_max=t_max, N=8, mode=rb.RADAR_STOCHASTIC, temperature=T, target_logits=tl, tree_tok=tok,
                               tree_parent=par, tree_draft_row=drow, n_nodes=n_nodes, retrieve=retrieve, n_leaves=n_leaves, draft_logits=dl,
                               R=2, u_accept=dev(u[None], np.float32), u_sample=dev([us], np.float32), accept_len=alen, path_nodes=nodes,
                               path_tokens=toks, next_token=nxt, best_retrieve_row=best, workspace=ws)
        ctx.check_device_status()
        assert nodes.cpu().tolist()[0] == path + [-1] * (t_max + 1 - len(path)) and int(alen) == len(path) - 1
        assert int(nxt) == int(np.searchsorted(cdf, float(us) * cdf[-1], side="right"))
    ctx.close()


def test_exponentials_to_the_last_places():
    """Two tokens that matter, q = 1/2 each: P_acc of the one d below the other is 2 e^-d / (1 + e^-d), to the 1.1 ulp of the
    exponential and half an ulp for each of the sum, two products and the quotient: below 4 units of 2^-53 x 2."""
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx, B, V = rb.Context(0), 2048, 5
    rng = np.random.default_rng(3)
    d = np.concatenate([rng.uniform(0, 2, B // 4), rng.uniform(0, 40, B // 4), rng.uniform(0, 700, B // 2)]).astype(np.float32)
    target, draft = np.full((B, 64, V), -np.inf, np.float32), np.full((B, 1, V), -np.inf, np.float32)
    target[:, 0, 1], target[:, 0, 3], draft[:, 0, 1], draft[:, 0, 3] = 0.0, -d, 0.5, 0.5
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    rows = lambda a, b, fill: dev(np.tile(np.array([[a, b] + [fill] * 62], np.int32), (B, 1)))
    dist, pacc = (torch.zeros(B, n, dtype=torch.float64, device="cuda") for n in (2, 64))
    ws = torch.zeros(rb.radar_acclen_workspace_bytes(ctx, B, V), dtype=torch.uint8, device="cuda")
    rb.radar_accept_length_distribution(ctx, B=B, V=V, t_max=1, temperature=1.0, target_logits=dev(target), tree_tok=rows(-1, 3, -1),
                                        tree_parent=rows(-1, 0, -1), tree_depth=rows(0, 1, 0), tree_draft_row=rows(0, -1, -1),
                                        n_nodes=dev(np.full(B, 2, np.int32)), draft_logits=dev(draft), R=1, dist=dist, p_acc_node=pacc, workspace=ws)
    ctx.check_device_status()
    e = np.exp(-d.astype(np.longdouble))
    want = np.minimum(2 * e / (1 + e), 1)
    assert np.max(np.abs(pacc[:, 1].cpu().numpy() / want - 1)) < 8 * 2.0 ** -53
    ctx.close()
