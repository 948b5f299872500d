"""Device buffers and the launch sequence of one speculative step.

`SpecStep` owns the torch tensors one step needs (pool, frontier, tree, attention output,
acceptance output, workspaces) and issues the library calls in order on the current
stream: t_max expansion calls (sequences the prediction model has stopped are skipped on
the device, so no decision ever returns to the host), rerank + tree build, tree
attention, acceptance.  Which form the expansion calls take is a matter of when their draft logits exist:

  `expand(t, ...)`, or `run_expansion(pipelined=False)`: one call behind the other.  The form of a decoding loop, whose
      draft model runs on the frontier of call t before the logits of call t + 1 are there.
  `run_expansion(pipelined=True)`: for logits that are all there before call 1 (recorded ones, gathering training data for
      the gate, a draft model that does not look at the frontier).  Several calls go in one go (`radar_expand_range`): all
      of them with short passes, a few at a time with long ones.  Batches too large for that, and features that do not lie
      in one piece, run as two overlapping chains: the bandwidth-bound vocabulary passes ahead on a side stream, the
      merge + select + gate kernels behind them on the main stream (the pass of call t+1 skips the sequences that had
      stopped before call t; one that stops at call t is read once in vain).

It contains no arithmetic of the method.
"""
from __future__ import annotations

import torch

from . import binding as rb


def _ranges(t_max, call_bytes):
    """The draft calls that are made in one go.  A range costs three launches, some 12 us; a call that is read and not
    made, its logits.  So with short passes (a call's rows of 24 MB take 4 us) up to eight calls go together, then up to
    four, and beyond 48 MB two and then about three at a time.  us for 1, 4, 5 to 7 and 8 calls, t_max = 8, V = 128256, k = 10:
        B = 4   two chains 29 / 58 / 83 / 89     8: 35 / 44 / 51 / 52     4, 4: 28 / 35 / 65 / 66     2, 3, 3: 24 / 52 / 74 / 77
        B = 8              38 / 74 / 101 / 114      55 / 64 / 71 / 73           41 / 48 / 85 / 87              32 / 67 / 86 / 99
        B = 32             91 / 200 / 278 / 318     195 / 204 / 212 / 212      117 / 124 / 221 / 220           79 / 155 / 210 / 231
    (two chains: the calls one by one, the passes ahead on a second stream, as they were before there were ranges)."""
    first = 0 if call_bytes <= 48 << 20 else 2
    most = 8 if call_bytes <= 24 << 20 else 4
    left = t_max - min(first, t_max)
    n = -(-left // most) if not first else max(round(left / 3), 1) if left else 0
    sizes = ([min(first, t_max)] if first else []) + [left // n + (i < left % n) for i in range(n)]
    ends = [sum(sizes[:i + 1]) for i in range(len(sizes))]
    return [(e - x + 1, e) for x, e in zip(sizes, ends)]


class SpecStep:
    def __init__(self, ctx: rb.Context, *, B, V, k, t_max, N, Hq, Hkv, d, kv_dtype, max_prefix_len,
                 mode=rb.RADAR_GREEDY, temperature=1.0, logits_dtype=torch.float32, device="cuda:0"):
        self.ctx = ctx
        self.B, self.V, self.k, self.t_max, self.N = B, V, k, t_max, N
        self.Hq, self.Hkv, self.d = Hq, Hkv, d
        self.kv_dtype, self.logits_dtype = kv_dtype, logits_dtype
        self.max_prefix_len = max_prefix_len
        self.mode, self.temperature = mode, float(temperature)
        self.C = k + (t_max - 1) * k * k
        self.R = 1 + (t_max - 1) * k
        dev = torch.device(device)
        self.dev = dev
        i32, f32, u8, i64 = torch.int32, torch.float32, torch.uint8, torch.int64
        z = lambda shape, dt: torch.zeros(shape, dtype=dt, device=dev)
        H, M = rb.RADAR_GATE_HIDDEN, rb.RADAR_MAX_NODES
        # expansion state
        self.active = z((B,), u8)
        self.cont = z((B,), u8)
        self.h, self.c = z((B, H), f32), z((B, H), f32)
        self.pool_tok, self.pool_parent = z((B, self.C), i32), z((B, self.C), i32)
        self.pool_depth, self.pool_draft_row = z((B, self.C), i32), z((B, self.C), i32)
        self.pool_score, self.pool_len = z((B, self.C), f32), z((B,), i32)
        self.root_score, self.root_pool_idx = z((B, 1), f32), torch.full((B, 1), -1, dtype=i32, device=dev)
        # per-call outputs, one slot per draft call so that a whole step can be inspected afterwards
        T = t_max
        self.frontier_tok, self.frontier_score = z((T, B, k), i32), z((T, B, k), f32)
        self.frontier_pool_idx, self.frontier_src_row = z((T, B, k), i32), z((T, B, k), i32)
        self.topk_tok, self.topk_logp = z((T, B, k, k), i32), z((T, B, k, k), f32)
        self.topk_tok1, self.topk_logp1 = z((B, 1, k), i32), z((B, 1, k), f32)      # call 1 has one row
        self.gate_logits, self.cont_hist = z((T, B, 2), f32), z((T, B), u8)
        # tree
        self.tree_tok, self.tree_parent, self.tree_depth = z((B, M), i32), z((B, M), i32), z((B, M), i32)
        self.tree_pos, self.tree_pool_idx, self.tree_draft_row = z((B, M), i32), z((B, M), i32), z((B, M), i32)
        self.tree_score, self.tree_mask = z((B, M), f32), z((B, M), i64)
        self.n_nodes, self.n_leaves = z((B,), i32), z((B,), i32)
        self.retrieve = z((B, N, t_max + 1), i32)
        # attention + acceptance outputs
        self.O = z((B, M, Hq, d), kv_dtype)
        self.lse = z((B, Hq, M), f32)
        self.accept_len, self.next_token, self.best_retrieve_row = z((B,), i32), z((B,), i32), z((B,), i32)
        self.path_nodes, self.path_tokens = z((B, t_max + 1), i32), z((B, t_max + 1), i32)
        # workspaces
        wb = max(rb.radar_expand_workspace_bytes(ctx, B, 1, V, k), rb.radar_expand_workspace_bytes(ctx, B, k, V, k))
        self.ws_expand = z((wb + 255,), u8)
        self.ws_expand2 = z((wb + 255,), u8)          # consecutive calls alternate, so a pass can run ahead of the select
        cb = rb.radar_expand_calls_workspace_bytes(ctx, B, V, k, t_max)
        self.ranges = [(1, t_max)] if cb else _ranges(t_max, B * k * V * logits_dtype.itemsize)
        sizes = [rb.radar_expand_range_workspace_bytes(ctx, B, V, k, *r) for r in self.ranges]
        cb = max(sizes) if min(sizes) else 0
        self.ws_calls = z((cb + 255,), u8) if cb else None      # None: the calls are issued one by one
        self.ws_attn = z((rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.dtype_code(self.O), max_prefix_len) + 255,), u8)
        self.ws_accept = z((rb.radar_accept_workspace_bytes(ctx, B, V, mode) + 255,), u8)
        self.side = torch.cuda.Stream(dev)            # the vocabulary passes of the pipelined expansion
        for n in ("ws_expand", "ws_expand2", "ws_attn", "ws_accept") + (("ws_calls",) if cb else ()):
            t = getattr(self, n)
            off = (-t.data_ptr()) % 256
            setattr(self, n, t[off:off + t.numel() - 255])

    # ---- expansion -------------------------------------------------------------------
    def _slots(self):
        """The addresses of the per-call outputs as one tuple per draft call: (frontier_tok, frontier_score, frontier_pool_idx,
        frontier_src_row, topk_tok, topk_logp, gate_logits, cont).  Worked out from the buffers each time a step is
        issued (indexing 64 views out of them instead costs 75 us a step of host time)."""
        f32, i32 = torch.float32, torch.int32
        bufs = ((self.frontier_tok, i32), (self.frontier_score, f32), (self.frontier_pool_idx, i32), (self.frontier_src_row, i32),
                (self.topk_tok, i32), (self.topk_logp, f32), (self.gate_logits, f32), (self.cont_hist, torch.uint8))
        return list(zip(*(range(p, p + x.numel() * x.element_size(), x.stride(0) * x.element_size())
                          for x, p in ((x, rb._ptr(x, dt)) for x, dt in bufs))))

    def expand(self, t, draft_logits, gate, force_calls=None, policy=rb.RADAR_POLICY_LSTM_SCORES, features=None,
               phase=rb.RADAR_EXPAND_ALL, vocab_mask=None, workspace=None, stream=None, slots=None):
        """Draft call t (1-based) on draft_logits [B,R,V]: row 0 for t = 1, rows 1+(t-2)k.. for t >= 2.
        `features` [t_max-1, B, feat_dim] feeds the hidden-state policy (row t-1 at call t).  `phase`, `vocab_mask`
        (the mask a RADAR_EXPAND_VOCAB call reads rows by), `workspace` and `stream` serve the pipelined form;
        `slots` is what `_slots()` returns, for callers that make several calls.  Returns the arguments of the call."""
        k, B, V = self.k, self.B, self.V
        F = 1 if t == 1 else k
        row0 = 0 if t == 1 else 1 + (t - 2) * k
        s = t - 1
        slots = self._slots() if slots is None else slots
        frontier_tok, frontier_score, frontier_pool_idx, frontier_src_row, topk_tok, topk_logp, gate_logits, cont = slots[s]
        kw = {
            "B": B, "F": F, "V": V, "k": k, "t": t, "t_max": self.t_max, "logits_row_stride": V, "logits_seq_stride": self.R * V,
            "parent_score": self.root_score if t == 1 else slots[s - 1][1],
            "parent_pool_idx": self.root_pool_idx if t == 1 else slots[s - 1][2],
            "active": vocab_mask if phase == rb.RADAR_EXPAND_VOCAB else self.active, "force_calls": force_calls, "h": self.h, "c": self.c,
            "pool_capacity": self.C, "pool_tok": self.pool_tok, "pool_parent": self.pool_parent, "pool_depth": self.pool_depth,
            "pool_draft_row": self.pool_draft_row, "pool_score": self.pool_score, "pool_len": self.pool_len,
            "frontier_tok": frontier_tok, "frontier_score": frontier_score, "frontier_pool_idx": frontier_pool_idx,
            "frontier_src_row": frontier_src_row, "topk_tok": self.topk_tok1 if t == 1 else topk_tok,
            "topk_logp": self.topk_logp1 if t == 1 else topk_logp, "gate_logits": gate_logits, "cont": cont, "policy": policy, "phase": phase}
        rb.expand_fields(self.ctx, kw, draft_logits, gate, self.ws_expand if workspace is None else workspace, row0 * V,
                         None if features is None or t >= self.t_max else features[s], stream)
        return kw

    def run_expansion(self, draft_logits, gate, force_calls=None, policy=rb.RADAR_POLICY_LSTM_SCORES, features=None,
                      pipelined=True):
        """All draft calls of a step on draft_logits [B,R,V].  `pipelined` needs the rows of all calls before the first one
        (see the top of this file); without it call t reads its own rows only."""
        together = self.ws_calls is not None
        if policy == rb.RADAR_POLICY_LSTM_HIDDEN and self.t_max > 1:          # all calls' features in one piece
            together = together and torch.is_tensor(features) and features.is_contiguous() and features.dim() == 3 and \
                features.shape[0] >= self.t_max - 1 and features.shape[1] == self.B
        if pipelined and together:
            self._expand_calls(draft_logits, gate, force_calls, policy, features)
            return
        slots = self._slots()
        if not pipelined:
            self._one_by_one(draft_logits, gate, force_calls, policy, features, slots)
            return
        # Two chains.  The vocabulary pass of call t (side stream, workspace t % 2) needs the select + gate block
        # of call t - 2 done: that block wrote the mask the pass skips rows by (cont of call t - 2; nothing for
        # t <= 2) and was the last reader of the same workspace.  The select + gate block of call t (main stream)
        # needs its pass and the block of call t - 1, which precedes it on the stream.
        main, side = torch.cuda.current_stream(), self.side
        ws = (self.ws_expand, self.ws_expand2)
        args = (draft_logits, gate, force_calls, policy, features)
        side.wait_stream(main)                      # fork: whatever produced the inputs is done
        sel_done = {}
        for t in range(1, self.t_max + 1):
            if t - 2 in sel_done:
                side.wait_event(sel_done[t - 2])
            mask = slots[t - 3][7] if t >= 3 else None
            self.expand(t, *args, phase=rb.RADAR_EXPAND_VOCAB, vocab_mask=mask, workspace=ws[t % 2], stream=side, slots=slots)
            voc = torch.cuda.Event()
            voc.record(side)
            main.wait_event(voc)
            self.expand(t, *args, phase=rb.RADAR_EXPAND_SELECT, workspace=ws[t % 2], stream=main, slots=slots)
            sel_done[t] = torch.cuda.Event()
            sel_done[t].record(main)
        main.wait_stream(side)                      # join (the last pass has been waited for already)

    def _one_by_one(self, draft_logits, gate, force_calls, policy, features, slots):
        """One call behind the other (call 1 restarts the state on the device).  The host is what bounds this form, so the
        arguments are put together once, and a call changes those that differ from the call before (a step of eight calls,
        attention and acceptance is issued in 93 us, with all arguments anew for every call in 110)."""
        kw = self.expand(1, draft_logits, gate, force_calls, policy, features, slots=slots)
        ctx, k, call_bytes = self.ctx, self.k, self.k * self.V * draft_logits.element_size()
        kw["F"], kw["logits"] = k, kw["logits"] + self.V * draft_logits.element_size() - call_bytes
        for t in range(2, self.t_max + 1):
            kw["t"], kw["logits"] = t, kw["logits"] + call_bytes
            _, kw["parent_score"], kw["parent_pool_idx"], _, _, _, _, _ = slots[t - 2]
            (kw["frontier_tok"], kw["frontier_score"], kw["frontier_pool_idx"], kw["frontier_src_row"], kw["topk_tok"], kw["topk_logp"],
             kw["gate_logits"], kw["cont"]) = slots[t - 1]
            if features is not None:
                kw["features"] = features[t - 1] if t < self.t_max else None
            rb.expand_again(ctx, kw)

    def _expand_calls(self, draft_logits, gate, force_calls, policy, features):
        more = self.t_max > 1
        kw = dict(
            B=self.B, V=self.V, k=self.k, t_max=self.t_max, logits=draft_logits, logits_row_stride=self.V,
            logits_seq_stride=self.R * self.V, parent_score=self.root_score, parent_pool_idx=self.root_pool_idx, active=self.active,
            force_calls=force_calls, gate=gate, h=self.h, c=self.c, pool_capacity=self.C, pool_tok=self.pool_tok,
            pool_parent=self.pool_parent, pool_depth=self.pool_depth, pool_draft_row=self.pool_draft_row, pool_score=self.pool_score,
            pool_len=self.pool_len, frontier_tok=self.frontier_tok, frontier_score=self.frontier_score,
            frontier_pool_idx=self.frontier_pool_idx, frontier_src_row=self.frontier_src_row, topk_tok=self.topk_tok1,
            topk_logp=self.topk_logp1, topk_tok_next=self.topk_tok[1:] if more else None,
            topk_logp_next=self.topk_logp[1:] if more else None, gate_logits=self.gate_logits, cont=self.cont_hist, policy=policy,
            workspace=self.ws_calls)
        if policy == rb.RADAR_POLICY_LSTM_HIDDEN and more:
            kw.update(features=features, feat_dim=features.shape[-1])
        for first, last in self.ranges:
            rb.radar_expand_range(self.ctx, t_first=first, t_last=last, **kw)

    # ---- tree, attention, acceptance ------------------------------------------------------
    def build_tree(self, root_tok, prefix_len, n_keep=None):
        rb.radar_rerank_build_tree(
            self.ctx, B=self.B, N=self.N, t_max=self.t_max, pool_capacity=self.C, pool_tok=self.pool_tok,
            pool_parent=self.pool_parent, pool_depth=self.pool_depth, pool_draft_row=self.pool_draft_row,
            pool_score=self.pool_score, pool_len=self.pool_len, n_keep=n_keep, root_tok=root_tok,
            prefix_len=prefix_len, tree_tok=self.tree_tok, tree_parent=self.tree_parent, tree_depth=self.tree_depth,
            tree_pos=self.tree_pos, tree_pool_idx=self.tree_pool_idx, tree_draft_row=self.tree_draft_row,
            tree_score=self.tree_score, tree_mask=self.tree_mask, n_nodes=self.n_nodes, retrieve=self.retrieve,
            n_leaves=self.n_leaves)

    def attention(self, Q, Kc, Vc, kv_start, prefix_len, Kt, Vt, mask=None, n_nodes=None, block_table=None, page_size=0):
        rb.radar_tree_attention(
            self.ctx, B=self.B, Hq=self.Hq, Hkv=self.Hkv, d=self.d, Q=Q, Kc=Kc, Vc=Vc, kv_start=kv_start,
            prefix_len=prefix_len, max_prefix_len=self.max_prefix_len, Kt=Kt, Vt=Vt,
            mask=self.tree_mask if mask is None else mask, n_nodes=self.n_nodes if n_nodes is None else n_nodes,
            O=self.O, lse=self.lse, workspace=self.ws_attn, block_table=block_table, page_size=page_size)

    def accept(self, target_logits, draft_logits=None, u_accept=None, u_sample=None):
        rb.radar_verify_accept(
            self.ctx, B=self.B, V=self.V, t_max=self.t_max, N=self.N, mode=self.mode, temperature=self.temperature,
            target_logits=target_logits, tree_tok=self.tree_tok, tree_parent=self.tree_parent,
            tree_draft_row=self.tree_draft_row, n_nodes=self.n_nodes, retrieve=self.retrieve, n_leaves=self.n_leaves,
            draft_logits=draft_logits, R=self.R, u_accept=u_accept, u_sample=u_sample, accept_len=self.accept_len,
            path_nodes=self.path_nodes, path_tokens=self.path_tokens, next_token=self.next_token,
            best_retrieve_row=self.best_retrieve_row, workspace=self.ws_accept)
