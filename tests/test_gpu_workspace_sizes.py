"""A workspace that was sized for the longest prefix, or the largest batch, serves the smaller ones."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,dtype", [(1, 4, 4, 64, "f32"), (1, 32, 8, 128, "f32"), (3, 1, 1, 128, "f32"), (1, 6, 2, 64, "bf16"), (2, 28, 4, 128, "bf16")])
def test_attention_with_shorter_prefixes(B, Hq, Hkv, d, dtype):
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx, longest = rb.Context(0), 4096
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    Q, Kt, Vt = (torch.randn(B, 64, h, d, device="cuda").to(dt) for h in (Hq, Hkv, Hkv))
    Kc, Vc = (torch.randn(B * longest, Hkv, d, device="cuda").to(dt) for _ in range(2))
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.dtype_code(Q), longest), dtype=torch.uint8, device="cuda")
    mask = torch.ones(B, 64, dtype=torch.int64, device="cuda")
    for P in list(range(0, 1200, 61)) + [960, 976, 1600, 2048, 2112, 3000, 4000, 4095, 4096]:
        lens = torch.full((B,), P, dtype=torch.int32, device="cuda")
        rb.radar_tree_attention(ctx, B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc[:max(1, B * P)], Vc=Vc[:max(1, B * P)], prefix_len=lens, max_prefix_len=P,
                                kv_start=torch.arange(B, device="cuda") * P, Kt=Kt, Vt=Vt, mask=mask, O=torch.empty_like(Q), workspace=ws,
                                n_nodes=torch.full((B,), 20, dtype=torch.int32, device="cuda"))
    ctx.check_device_status()
    ctx.close()
