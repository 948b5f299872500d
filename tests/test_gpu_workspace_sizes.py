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


@pytest.mark.parametrize("largest,V,k", [(34, 8000, 10), (80, 8192, 4), (6, 16000, 32), (20, 50257, 8), (160, 4000, 2)])
def test_expansion_and_greedy_acceptance_of_smaller_batches(largest, V, k):
    """The vocabulary pass cuts a row into smaller chunks where there are few rows: a smaller batch may need more records."""
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    from paper_2512_14069_b200 import workloads as W
    ctx, t_max = rb.Context(0), 3
    gate = {n: torch.from_numpy(w).cuda() for n, w in W.gate_weights(W.shrink(W.CONFIGS[2], k=k)).items()}
    step = lambda B: SpecStep(ctx, B=B, V=V, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
    big = step(largest)
    draft = torch.randn(largest, big.R, V, device="cuda")
    target = torch.randn(largest, 64, V, device="cuda")
    calls_ws = rb.radar_expand_calls_workspace_bytes(ctx, largest, V, k, t_max)
    for B in sorted({b for b in (1, 2, 3, 4, 5, largest // 4, largest // 3, largest // 2, 29, 36, 73, largest - 1, largest) if 0 < b <= largest}):
        s = step(B)
        s.ws_expand, s.ws_expand2, s.ws_accept = big.ws_expand, big.ws_expand2, big.ws_accept
        s.run_expansion(draft[:B].contiguous(), gate, pipelined=False)
        if calls_ws and s.ws_calls is not None:
            assert rb.radar_expand_calls_workspace_bytes(ctx, B, V, k, t_max) <= calls_ws
        s.build_tree(torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda"))
        s.accept(target[:B].contiguous())
        ctx.check_device_status()
        n = s.n_nodes.cpu()
        first = [int(target[b, 0].argmax()) for b in range(B)]
        assert all(int(s.next_token[b]) == first[b] for b in range(B) if int(s.accept_len[b]) == 0) and int(n.min()) > 0
    ctx.close()
