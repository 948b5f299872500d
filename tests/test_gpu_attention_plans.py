"""Grid plans of the tensor-core attention that depend on the number of layers and on there being one sequence: units of
two row blocks across many layers, and grids in which every CTA has one piece of one unit.  Against the oracle, over
prefix lengths at tile edges; tolerance of the bf16 path (2e-2 max-abs: bf16 P and O)."""
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


@pytest.mark.parametrize("P,Hq,Hkv", [(1, 8, 8), (511, 8, 2), (512, 8, 2), (513, 8, 2), (1025, 4, 4), (3000, 28, 4), (2100, 32, 1)])
def test_one_sequence(ctx, P, Hq, Hkv):
    cfg = W.shrink(W.CONFIGS[5], cid=400 + Hq, B=1, Hq=Hq, Hkv=Hkv, P=(P, P), V=2000, k=4, t_max=5, N=63)
    inp = H.make_inputs(cfg)
    _, _, trees = H.oracle_expand_and_tree(cfg, inp)
    g = H.CudaRun(cfg, inp, ctx)
    g.upload_attention()
    O_gpu, lse_gpu = g.attention(trees)
    O_ref, lse_ref = H.oracle_attention(cfg, inp, trees)
    H.compare_attention(cfg, O_gpu, lse_gpu, O_ref, lse_ref, trees)


@pytest.mark.parametrize("L,P,Hq,Hkv", [(2, 700, 8, 8), (48, 700, 8, 2), (90, 600, 4, 1)])
def test_many_layers_of_one_sequence(ctx, L, P, Hq, Hkv):
    import torch
    from paper_2512_14069_b200 import binding as rb
    cfg = W.shrink(W.CONFIGS[5], cid=420 + L, B=1, Hq=Hq, Hkv=Hkv, P=(P, P), V=2000, k=4, t_max=5, N=60)
    inp = H.make_inputs(cfg)
    _, _, trees = H.oracle_expand_and_tree(cfg, inp)
    rng = np.random.default_rng(L)
    sign = torch.from_numpy(rng.choice([-1.0, 1.0], size=L).astype(np.float32)).cuda().to(torch.bfloat16)
    Q, Kt, Vt, Kc, Vc = (H.to_dev(np.stack(inp[n]) if n in ("Kc", "Vc") else inp[n]) for n in ("Q", "Kt", "Vt", "Kc", "Vc"))
    # layer l: values times +-1 and the heads rolled by l, so that a mix-up of layers or heads shows
    roll = lambda x, l, heads: torch.roll(x, shifts=l % heads, dims=-2)
    QL = torch.stack([roll(Q, l * (Hq // Hkv), Hq) for l in range(L)])
    KtL, KcL = (torch.stack([roll(x, l, Hkv) for l in range(L)]).contiguous() for x in (Kt, Kc[0]))
    VtL, VcL = (torch.stack([roll(x, l, Hkv) * sign[l] for l in range(L)]).contiguous() for x in (Vt, Vc[0]))
    mask = H.to_dev(np.stack([t["mask"] for t in trees]).view(np.int64))
    n_nodes = H.to_dev(np.array([t["n_nodes"] for t in trees], np.int32))
    O, lse = torch.zeros_like(QL), torch.zeros(L, 1, Hq, 64, device="cuda")
    wb = rb.radar_attn_workspace_bytes(ctx, 1, Hq, Hkv, cfg.d, rb.RADAR_BF16, P)
    ws = torch.zeros(wb, dtype=torch.uint8, device="cuda")
    rb.radar_tree_attention(ctx, B=1, Hq=Hq, Hkv=Hkv, d=cfg.d, Q=QL, Kc=KcL, Vc=VcL, kv_start=torch.zeros(1, dtype=torch.int64, device="cuda"),
                            prefix_len=H.to_dev(inp["prefix_len"]), max_prefix_len=P, Kt=KtL, Vt=VtL, mask=mask, n_nodes=n_nodes, O=O,
                            lse=lse, workspace=ws, n_layers=L)
    ctx.check_device_status()
    O_ref, lse_ref = H.oracle_attention(cfg, inp, trees)
    n = trees[0]["n_nodes"]
    for l in range(L):
        back = torch.roll(O[l], shifts=-(l * (Hq // Hkv)) % Hq, dims=-2).float() * float(sign[l])
        lback = torch.roll(lse[l], shifts=-(l * (Hq // Hkv)) % Hq, dims=-2)
        H.compare_attention(cfg, back.cpu().numpy(), lback.cpu().numpy(), O_ref, lse_ref, trees)
        assert not O[l, :, n:].any()
