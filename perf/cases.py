"""The timed cases: what users of this library have it do, over the sizes they do it at.

Four kinds of work:

step     one speculative step through `SpecStep`: t_max draft calls with the gate, rerank + tree, one layer of tree
         attention, acceptance.  Serving loops capture the step in a CUDA graph (as bench.py does) and replay it; where
         the draft model runs between the calls, the loop issues them one at a time.
layers   the verification pass of a whole target model: the attention of all its layers in one call.
acclen   acceptance-length distributions (Eq. 11-13) of verified trees: how training data for the gate is gathered.
train    one REINFORCE step of the prediction model.
"""
import math

import numpy as np
import torch

from paper_2512_14069_b200 import binding as rb
from paper_2512_14069_b200 import workloads as W
from paper_2512_14069_b200.pipeline import SpecStep

_DT = {"f32": torch.float32, "bf16": torch.bfloat16}
_H, _M = rb.RADAR_GATE_HIDDEN, rb.RADAR_MAX_NODES
_HYPER = dict(alpha=0.05, gamma=0.99, T_o=68.0, T_d=2.7, T_p=0.4)     # training terms, LLaMA-3.1-8B in the paper
_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = rb.Context(torch.cuda.current_device())
    return _ctx


# calls_lo / calls_hi: draft calls of a sequence, drawn per sequence (a trained gate stops after 5 to 7 on average);
# 0: the gate of configuration `gate_cfg` decides, whose bias puts the stop inside the trajectory.
_STEP = dict(kind="step", B=1, V=128256, k=10, t_max=8, N=60, keep_lo=60, Hq=32, Hkv=8, d=128, kv="bf16", logits="f32",
             P_lo=2048, P_hi=2048, page=0, mode="greedy", temperature=1.0, peak_lo=1.0, peak_hi=1.0, sigma=1.0, calls_lo=0,
             calls_hi=0, gate_cfg=2, policy="lstm", feat_dim=0, graph=True, pipelined=True)


def listed():
    def s(name, **kw):
        return dict(_STEP, name=name, **kw)
    return [
        # the smallest call: one short request, small vocabulary, everything in fp32
        s("step_tiny_f32", V=1000, k=4, t_max=4, N=16, keep_lo=16, Hq=4, Hkv=4, d=64, kv="f32", P_lo=128, P_hi=128, sigma=0.5,
          gate_cfg=1),
        # interactive decoding of one request on an 8B model: latency of a chain of small kernels
        s("step_8b_b1"),
        # the same model behind a draft model that runs between the calls: nothing captured, nothing runs ahead
        s("step_8b_b1_call_by_call", P_lo=3001, P_hi=3001, calls_lo=6, calls_hi=6, graph=False, pipelined=False),
        # multi-head attention, small batch, sampling at T = 1, logits of differing peakedness
        s("step_13b_b4", B=4, V=32000, k=8, t_max=6, N=48, keep_lo=48, Hq=40, Hkv=40, P_lo=4096, P_hi=4096, mode="stochastic",
          peak_lo=0.5, peak_hi=2.0, gate_cfg=3),
        # a 70B model's layer, ragged trees, greedy
        s("step_70b_b8", B=8, Hq=64, Hkv=8, P_lo=8192, P_hi=8192, calls_lo=1, calls_hi=8),
        # a server under load: 32 ragged requests with long contexts, sampling
        s("step_8b_b32", B=32, P_lo=4096, P_hi=32768, mode="stochastic", temperature=0.7, keep_lo=8, calls_lo=2, calls_hi=8),
        # a server with bf16 logits and a paged cache, three query heads per KV head, a vocabulary that aligns to nothing
        s("step_gqa3_b6_paged", B=6, V=50257, k=6, t_max=6, N=31, keep_lo=20, Hq=24, Hkv=8, logits="bf16", P_lo=300, P_hi=4500,
          page=16, mode="stochastic", temperature=0.9, calls_lo=3, calls_hi=6),
        # all layers of an 8B model's verification pass for one request
        dict(kind="layers", name="layers_8b_b1", B=1, L=32, Hq=32, Hkv=8, d=128, P_lo=2048, P_hi=2048, page=0, N=60, calls=6),
        # ... and of 32 layers at a 70B model's shapes, ragged contexts
        dict(kind="layers", name="layers_70b_b8", B=8, L=32, Hq=64, Hkv=8, d=128, P_lo=6000, P_hi=8192, page=0, N=60, calls=6),
        # training data for the gate: four Vicuna-13B trees, and eight with the large vocabulary
        dict(kind="acclen", name="acclen_13b_b4", B=4, V=32000, k=8, t_max=6, N=48, calls=6, logits="f32", temperature=1.0),
        dict(kind="acclen", name="acclen_8b_b8", B=8, V=128256, k=10, t_max=8, N=60, calls=5, logits="f32", temperature=1.0),
        # the paper's batch of 256 data points
        dict(kind="train", name="train_256", n=256, k=10, t_max=8),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choices(["step", "layers", "acclen", "train"], [0.64, 0.12, 0.12, 0.12])[0]
    heads = [(4, 4), (16, 16), (40, 40), (32, 8), (64, 8), (24, 8), (28, 4), (32, 4), (16, 1)]
    if kind == "train":
        return dict(kind=kind, n=log_int(1, 1024), k=rng.randint(1, 16), t_max=rng.randint(2, 10))
    if kind == "acclen":
        t_max = rng.randint(2, 8)
        V = log_int(1000, 152000)
        return dict(kind=kind, B=log_int(1, max(1, min(16, 1000000 // V))), V=V, k=rng.randint(2, 12), t_max=t_max, N=rng.randint(8, 63),
                    calls=rng.randint(1, t_max), logits=rng.choice(["f32", "bf16"]), temperature=rng.choice([0.7, 1.0, 1.3]))
    Hq, Hkv = rng.choice(heads)
    d = rng.choice([64, 128, 128])
    page = rng.choice([0, 0, 0, 16, 64, 128])
    if kind == "layers":
        L = log_int(2, 32)
        B = log_int(1, 8)
        P_hi = log_int(64, min(16384, 8.0e9 // (L * B * Hkv * d * 4)))
        return dict(kind=kind, B=B, L=L, Hq=Hq, Hkv=Hkv, d=d, P_lo=rng.randint(max(1, P_hi // 4), P_hi), P_hi=P_hi, page=page,
                    N=rng.randint(16, 63), calls=rng.randint(2, 7))
    t_max = rng.randint(2, 8)
    k = rng.choice([1, 2, 4, 6, 8, 10, 10, 12, 16])
    logits = rng.choice(["f32", "f32", "bf16"])
    V = log_int(1000, 152000)
    rows = 1 + (t_max - 1) * k + _M
    B = log_int(1, max(1, min(32, 4.4e8 // (rows * V))))
    kv = "f32" if B <= 2 and rng.random() < 0.2 else "bf16"
    P_hi = log_int(16, max(16, min(32768, 2.0e9 // (B * Hkv * d * 4), 2048 if kv == "f32" else 32768)))
    N = rng.randint(8, 63)
    policy = rng.choice(["lstm"] * 8 + ["mlp", "hidden"])
    calls = rng.randint(1, t_max)
    graph = rng.random() < 0.8
    return dict(_STEP, B=B, V=V, k=k, t_max=t_max, N=N, keep_lo=rng.choice([N, max(1, N // 3)]), Hq=Hq, Hkv=Hkv, d=d, kv=kv,
                logits=logits, P_lo=rng.randint(max(1, P_hi // 4), P_hi), P_hi=P_hi, page=page,
                mode=rng.choice(["greedy", "stochastic"]), temperature=rng.choice([0.7, 1.0]), peak_lo=rng.choice([0.5, 1.0]),
                peak_hi=rng.choice([1.0, 2.0]), calls_lo=calls, calls_hi=rng.randint(calls, t_max), gate_cfg=2, policy=policy,
                feat_dim=rng.choice([64, 1000, 4096]) if policy == "hidden" else 0, graph=graph, pipelined=graph or rng.random() < 0.3)


# ---- inputs ------------------------------------------------------------------------------------------------------
def _peaked_rows(g, n, V, a, dtype):
    """[n, V] logits whose sorted values fall off as -a ln(rank), like a language model's."""
    z = torch.rand(n, V, device="cuda", generator=g).mul_(V).log1p_().mul_(-a)
    return z.add_(torch.randn(n, V, device="cuda", generator=g), alpha=0.1).to(dtype)


def _target_rows(g, draft, draft_row, a, sigma, dtype):
    """[64, V] target logits of one tree: the draft row behind each node (a fresh row where there is none) plus noise."""
    V = draft.shape[-1]
    t = _peaked_rows(g, _M, V, a, torch.float32)
    has = draft_row >= 0
    t[has] = draft[draft_row[has].long()].float()
    return t.add_(torch.randn(_M, V, device="cuda", generator=g), alpha=sigma).to(dtype)


def _ints(rng, lo, hi, n):
    return torch.from_numpy(rng.integers(lo, hi + 1, size=n).astype(np.int32)).cuda()


def _grown_trees(c, rng, g, logits="f32", V=4096, k=10, t_max=8, peak=(1.0, 1.0)):
    """A SpecStep whose trees have been built from `calls` draft calls, and the draft logits behind them."""
    B = c["B"]
    step = SpecStep(_context(), B=B, V=V, k=k, t_max=t_max, N=c["N"], Hq=c.get("Hq", 4), Hkv=c.get("Hkv", 4), d=c.get("d", 64),
                    kv_dtype=torch.bfloat16, max_prefix_len=c.get("P_hi", 1), logits_dtype=_DT[logits])
    draft = torch.empty(B, step.R, V, device="cuda", dtype=_DT[logits])
    a = rng.uniform(*peak, size=B)
    for b in range(B):
        draft[b] = _peaked_rows(g, step.R, V, float(a[b]), _DT[logits])
    gate = {n: torch.from_numpy(w).cuda() for n, w in W.gate_weights(W.shrink(W.CONFIGS[2], k=k)).items()}
    plen = _ints(rng, c.get("P_lo", 1), c.get("P_hi", 1), B)
    force = torch.full((B,), c["calls"], dtype=torch.int32, device="cuda")
    step.run_expansion(draft, gate, force)
    step.build_tree(_ints(rng, 0, V - 1, B), plen)
    return step, draft, plen, a


def _cache(c, plen, g, layers=None):
    """Keys and values of the prefixes: rows of all sequences packed, or in pages scattered by a block table."""
    lens = plen.cpu().numpy().astype(np.int64)
    if c["page"]:
        pages = -(-lens // c["page"])
        perm = torch.randperm(int(pages.sum()), device="cuda", generator=g).to(torch.int32)
        table = torch.zeros(len(lens), -(-c["P_hi"] // c["page"]), dtype=torch.int32, device="cuda")
        at = 0
        for b, n in enumerate(pages):
            table[b, :n] = perm[at:at + n]
            at += int(n)
        rows, start = int(pages.sum()) * c["page"], None
    else:
        rows, table = int(lens.sum()), None
        start = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)[:-1]])).cuda()
    shape = (rows, c["Hkv"], c["d"]) if layers is None else (layers, rows, c["Hkv"], c["d"])
    dt = _DT[c.get("kv", "bf16")]
    K, V = (torch.randn(shape, device="cuda", generator=g, dtype=dt) for _ in range(2))
    return K, V, start, table


def _prepare_step(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    B, V, k, t_max = c["B"], c["V"], c["k"], c["t_max"]
    ldt, kdt = _DT[c["logits"]], _DT[c["kv"]]
    greedy = c["mode"] == "greedy"
    step = SpecStep(_context(), B=B, V=V, k=k, t_max=t_max, N=c["N"], Hq=c["Hq"], Hkv=c["Hkv"], d=c["d"], kv_dtype=kdt,
                    max_prefix_len=c["P_hi"], mode=rb.RADAR_GREEDY if greedy else rb.RADAR_STOCHASTIC, temperature=c["temperature"],
                    logits_dtype=ldt)
    a = rng.uniform(c["peak_lo"], c["peak_hi"], size=B)
    draft = torch.empty(B, step.R, V, device="cuda", dtype=ldt)
    for b in range(B):
        draft[b] = _peaked_rows(g, step.R, V, float(a[b]), ldt)
    cfg = W.shrink(W.CONFIGS[c["gate_cfg"]], k=k, t_max=t_max)
    features = None
    if c["policy"] == "lstm":
        w, policy = W.gate_weights(cfg), rb.RADAR_POLICY_LSTM_SCORES
    elif c["policy"] == "mlp":
        w, policy = W.policy_weights(cfg, "mlp_scores"), rb.RADAR_POLICY_MLP_SCORES
    else:
        w, policy = W.policy_weights(cfg, "lstm_hidden", c["feat_dim"]), rb.RADAR_POLICY_LSTM_HIDDEN
        features = torch.randn(max(t_max - 1, 1), B, c["feat_dim"], device="cuda", generator=g)
    gate = {n: torch.from_numpy(x).cuda() for n, x in w.items()}
    force = _ints(rng, c["calls_lo"], c["calls_hi"], B) if c["calls_lo"] else None
    keep, root = _ints(rng, c["keep_lo"], c["N"], B), _ints(rng, 0, V - 1, B)
    plen = _ints(rng, c["P_lo"], c["P_hi"], B)
    Kc, Vc, start, table = _cache(c, plen, g)
    Q = torch.randn(B, _M, c["Hq"], c["d"], device="cuda", generator=g, dtype=kdt)
    Kt, Vt = (torch.randn(B, _M, c["Hkv"], c["d"], device="cuda", generator=g, dtype=kdt) for _ in range(2))
    u_acc, u_smp = torch.rand(B, _M, device="cuda", generator=g), torch.rand(B, device="cuda", generator=g)

    def expand_and_build():
        step.run_expansion(draft, gate, force, policy, features, pipelined=c["pipelined"])
        step.build_tree(root, plen, keep)

    expand_and_build()                                # the target model's logits belong to the nodes of this tree
    target = torch.empty(B, _M, V, device="cuda", dtype=ldt)
    for b in range(B):
        target[b] = _target_rows(g, draft[b], step.tree_draft_row[b], float(a[b]), c["sigma"], ldt)

    def one_step():
        expand_and_build()
        step.attention(Q, Kc, Vc, start, plen, Kt, Vt, block_table=table, page_size=c["page"])
        if greedy:
            step.accept(target)
        else:
            step.accept(target, draft, u_acc, u_smp)

    replay = None
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            one_step()
            side.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                one_step()
        torch.cuda.current_stream().wait_stream(side)
        replay = graph.replay
    names = ("pool_tok", "pool_parent", "pool_depth", "pool_draft_row", "pool_score", "pool_len", "frontier_tok", "frontier_score",
             "frontier_pool_idx", "frontier_src_row", "topk_tok", "topk_logp", "topk_tok1", "topk_logp1", "gate_logits", "cont_hist",
             "h", "c", "active", "tree_tok", "tree_parent", "tree_depth", "tree_pos", "tree_pool_idx", "tree_draft_row", "tree_score",
             "tree_mask", "n_nodes", "retrieve", "n_leaves", "O", "lse", "accept_len", "path_nodes", "path_tokens", "next_token",
             "best_retrieve_row")
    # (one_step holds every tensor that the graph reads)
    return {"run": replay or one_step, "step": one_step, "out": {n: getattr(step, n) for n in names}}


def _prepare_layers(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    step, _, plen, _ = _grown_trees(c, rng, g)
    B, L, Hq, Hkv, d = c["B"], c["L"], c["Hq"], c["Hkv"], c["d"]
    Kc, Vc, start, table = _cache(c, plen, g, layers=L)
    Q = torch.randn(L, B, _M, Hq, d, device="cuda", generator=g, dtype=torch.bfloat16)
    Kt, Vt = (torch.randn(L, B, _M, Hkv, d, device="cuda", generator=g, dtype=torch.bfloat16) for _ in range(2))
    O, lse = torch.zeros_like(Q), torch.zeros(L, B, Hq, _M, device="cuda")

    def run():
        rb.radar_tree_attention(_context(), B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, kv_start=start, prefix_len=plen,
                                max_prefix_len=c["P_hi"], Kt=Kt, Vt=Vt, mask=step.tree_mask, n_nodes=step.n_nodes, O=O, lse=lse,
                                workspace=step.ws_attn, n_layers=L, block_table=table, page_size=c["page"])
    return {"run": run, "out": {"O": O, "lse": lse}}


def _prepare_acclen(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    B, V, t_max = c["B"], c["V"], c["t_max"]
    step, draft, _, a = _grown_trees(c, rng, g, c["logits"], V, c["k"], t_max, (0.5, 2.0))
    target = torch.empty(B, _M, V, device="cuda", dtype=_DT[c["logits"]])
    for b in range(B):
        target[b] = _target_rows(g, draft[b], step.tree_draft_row[b], float(a[b]), 1.0, _DT[c["logits"]])
    dist = torch.zeros(B, t_max + 1, device="cuda", dtype=torch.float64)
    p_acc = torch.zeros(B, _M, device="cuda", dtype=torch.float64)
    ws = torch.zeros(rb.radar_acclen_workspace_bytes(_context(), B, V), device="cuda", dtype=torch.uint8)

    def run():
        rb.radar_accept_length_distribution(
            _context(), B=B, V=V, t_max=t_max, temperature=c["temperature"], target_logits=target, tree_tok=step.tree_tok,
            tree_parent=step.tree_parent, tree_depth=step.tree_depth, tree_draft_row=step.tree_draft_row, n_nodes=step.n_nodes,
            draft_logits=draft, R=step.R, dist=dist, p_acc_node=p_acc, workspace=ws)
    return {"run": run, "out": {"dist": dist, "p_acc_node": p_acc}}


def _prepare_train(c, seed):
    n, k, t_max = c["n"], c["k"], c["t_max"]
    cfg = W.shrink(W.CONFIGS[2], k=k, t_max=t_max)
    log_states, dists, u_action, u_length = (torch.from_numpy(x).cuda() for x in W.train_batch(cfg, n, seed))
    w = W.gate_weights(cfg)
    theta = torch.from_numpy(np.concatenate([w[x].reshape(-1) for x in ("w_ih", "w_hh", "b_ih", "b_hh", "w1", "b1", "w2", "b2")])).cuda()
    m, v, grad = (torch.zeros_like(theta) for _ in range(3))
    loss = torch.zeros(1, device="cuda")
    calls, l_acc = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    actions = torch.zeros(n, t_max, dtype=torch.uint8, device="cuda")
    ws = torch.zeros(rb.radar_train_workspace_bytes(_context(), n, k, t_max), device="cuda", dtype=torch.uint8)
    done = [0]

    def run():
        done[0] += 1
        rb.radar_policy_train_step(_context(), n=n, k=k, t_max=t_max, log_states=log_states, dists=dists, u_action=u_action,
                                   u_length=u_length, theta=theta, grad=grad, loss=loss, calls=calls, l_acc=l_acc, actions=actions,
                                   workspace=ws, step=done[0], lr=1e-4, adam_m=m, adam_v=v, **_HYPER)
    return {"run": run, "out": {"theta": theta, "m": m, "v": v, "grad": grad, "loss": loss, "calls": calls, "l_acc": l_acc,
                                "actions": actions}}


def prepare(case, seed):
    return {"step": _prepare_step, "layers": _prepare_layers, "acclen": _prepare_acclen, "train": _prepare_train}[case["kind"]](case, seed)


def run(state):
    state["run"]()
    return state["out"]


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
def _tree_rows(c, calls):
    return min((c["N"] + c.get("keep_lo", c["N"])) / 2, c.get("k", 10) * (1 + (calls - 1) * c.get("k", 10))) + 1


def _attention(c, rows, e):
    P = (c["P_lo"] + c["P_hi"]) / 2
    n = c["B"] * c.get("L", 1)
    return (n * ((P + rows) * c["Hkv"] * c["d"] * 2 * e + 2 * rows * c["Hq"] * c["d"] * e),
            4.0 * n * rows * c["Hq"] * (P + rows) * c["d"])


def work(case):
    c = case
    if c["kind"] == "layers":
        b, f = _attention(c, _tree_rows(c, c["calls"]), 2)
        return {"bytes": b, "flops": f}
    if c["kind"] == "train":
        params = 4 * _H * (c["k"] + _H + 2) + _H * (_H + c["k"] + 1) + 2 * _H + 2
        data = c["n"] * (c["t_max"] * (c["k"] * 4 + (c["t_max"] + 1) * 8 + 5) + 12)
        return {"bytes": params * 7 * 4 + data, "flops": 6.0 * params * c["n"] * min(2.0, c["t_max"] - 1)}   # about two calls a rollout
    s = 2 if c["logits"] == "bf16" else 4
    if c["kind"] == "acclen":
        inner = min(1 + (c["calls"] - 1) * c["k"], _tree_rows(c, c["calls"]) / 2.5)           # rows with children
        return {"bytes": c["B"] * inner * 2 * c["V"] * s, "flops": c["B"] * inner * c["V"] * 30.0}
    calls = (c["calls_lo"] + c["calls_hi"]) / 2 or {1: 3, 2: 5, 3: 4.25}[c["gate_cfg"]]
    rows = _tree_rows(c, calls)
    b, f = _attention(c, rows, 2 if c["kv"] == "bf16" else 4)
    b += c["B"] * (1 + (calls - 1) * c["k"]) * c["V"] * s                                     # draft logits
    b += c["B"] * (rows if c["mode"] == "greedy" else 4) * c["V"] * s                         # target (and draft) rows of the walk
    b += 4 * (4 * _H * (c["k"] + _H + 2) + _H * (_H + c["k"] + 3))                              # the gate's weights
    b += c["feat_dim"] * 4 * (5 * _H + c["B"] * (calls - 1))
    return {"bytes": b, "flops": f}


def tolerance(case):
    # whole values (tokens, trees, paths) stay the same everywhere
    if case["kind"] == "acclen":
        return {"rel": 1e-9}                         # fp64 throughout
    if case["kind"] == "train":
        return {"rel": 2e-5, "max": 2e-3}            # fp32 sums in the gradients
    if case["kind"] == "step" and case["kv"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}            # fp32 sums; scores near zero
    return {"rel": 9e-3, "max": 0.05}                # bf16 attention: 2.3e-3 and 0.011 against the same sums in fp64
