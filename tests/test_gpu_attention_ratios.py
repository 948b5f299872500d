"""Tensor-core attention at head ratios that do not divide 128: a row block then holds 128 // G whole nodes and its last
128 % G rows are idle.  Against the oracle, at both plans (one and two row blocks per unit), over row-block edges, with
the pieces of cut units merged, in both cache layouts.  Tolerance of the bf16 path: 2e-2 max-abs (bf16 O;
the precision of P has a test of its own)."""
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


@pytest.mark.parametrize("Hq,Hkv,d,page,max_p", [
    (24, 8, 128, 0, None), (28, 4, 128, 0, None), (28, 4, 64, 16, None), (5, 1, 64, 0, None), (12, 1, 128, 0, 40000),
    (28, 4, 128, 0, 20000), (48, 1, 128, 0, 40000), (100, 1, 64, 0, 40000), (15, 3, 128, 128, None)])
def test_attention_ratio_not_dividing_128(ctx, Hq, Hkv, d, page, max_p):
    from paper_2512_14069_b200 import binding as rb
    cfg = W.shrink(W.CONFIGS[5], cid=300 + Hq + d + page, B=4, Hq=Hq, Hkv=Hkv, d=d, P=(400, 1100), V=2000, k=4, t_max=5, N=63)
    inp = H.make_inputs(cfg)
    _, _, trees = H.oracle_expand_and_tree(cfg, inp)
    per = 128 // (Hq // Hkv)                                            # nodes of a full row block
    trees[0] = dict(trees[0]); trees[0]["n_nodes"] = 1
    trees[1] = dict(trees[1]); trees[1]["n_nodes"] = min(per, int(trees[1]["n_nodes"]))          # exactly one row block
    trees[2] = dict(trees[2]); trees[2]["n_nodes"] = min(per + 1, int(trees[2]["n_nodes"]))      # one node in the next
    g = H.CudaRun(cfg, inp, ctx, max_prefix_len=max_p) if max_p else H.CudaRun(cfg, inp, ctx)
    g.upload_attention(page_size=page) if page else g.upload_attention()
    s = g.step
    path = rb.radar_tree_attention_path(B=cfg.B, Hq=Hq, Hkv=Hkv, d=d, Q=g.Q, Kc=g.Kc, Vc=g.Vc, kv_start=None if page else g.kv_start,
                                        prefix_len=g.prefix_len, max_prefix_len=s.max_prefix_len, Kt=g.Kt, Vt=g.Vt,
                                        mask=s.tree_mask, n_nodes=s.n_nodes, O=s.O, workspace=s.ws_attn)
    assert path == rb.RADAR_ATTN_PATH_TENSOR_CORE
    O_gpu, lse_gpu = g.attention(trees)
    ctx.check_device_status()
    O_ref, lse_ref = H.oracle_attention(cfg, inp, trees)
    H.compare_attention(cfg, O_gpu, lse_gpu, O_ref, lse_ref, trees)
