"""bf16 attention at head ratios that do not divide 128 keeps 32-bit probabilities: against fp64, all that is left is the rounding
of O to bf16.  One and two row blocks a unit, units in one piece, cut into a few and into many, both cache layouts, partial
last tiles, a tree tile alone.

Bounds: the probabilities are a sum of two bf16 numbers (2^-18 relative) and the sums fp32, which adds less than 1e-3 of the
rounding of O to bf16 (2^-9) to the 2-norm of its error; a single bf16 a probability would add 30 %.  lse: fp32 scores and
sums, 4 units in the last place of values up to 12."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,P,page,M", [
    (1, 24, 8, 128, 2048, 0, 61), (2, 28, 4, 128, 700, 16, 64), (3, 12, 4, 64, 333, 0, 20), (1, 12, 1, 128, 20000, 0, 60), (1, 28, 4, 64, 9000, 128, 33),
    (2, 100, 1, 64, 2000, 0, 64), (1, 40, 8, 128, 1400, 0, 64), (4, 24, 8, 128, 0, 0, 64), (8, 28, 4, 128, 3000, 0, 64),
    # little work: the FMA kernel, up to its line and one key above it
    (2, 6, 2, 64, 100, 0, 64), (1, 24, 8, 64, 100, 16, 30), (1, 3, 1, 128, 500, 0, 64), (1, 3, 1, 64, 1472, 0, 40), (1, 3, 1, 64, 1473, 0, 40)])
def test_probabilities_keep_32_bits(B, Hq, Hkv, d, P, page, M):
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx = rb.Context(0)
    g = torch.Generator(device="cuda").manual_seed(Hq * P + M)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    plen = torch.tensor([max(0, P - 37 * b) for b in range(B)], dtype=torch.int32)
    Q, Kt, Vt = rand(B, 64, Hq, d), rand(B, 64, Hkv, d), rand(B, 64, Hkv, d)
    start = torch.cumsum(plen.long(), 0) - plen
    table = None
    if page:
        pages = (plen + page - 1) // page
        first = torch.cumsum(pages, 0) - pages
        table = (first[:, None] + torch.arange(int(pages.max()))).to(torch.int32).cuda()
        start, n_rows = first.long() * page, int(pages.sum()) * page
    else:
        n_rows = max(int(plen.sum()), 1)
    Kc, Vc = rand(n_rows, Hkv, d), rand(n_rows, Hkv, d)
    low = torch.tril(torch.rand(B, 64, 64, device="cuda", generator=g) < 0.5) | torch.eye(64, device="cuda", dtype=torch.bool)
    low[:, :, 0] = True
    bits = (low.long() << torch.arange(64, device="cuda")).sum(-1)
    O, lse = torch.zeros_like(Q), torch.zeros(B, Hq, 64, device="cuda")
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.RADAR_BF16, P) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    kw = dict(B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, kv_start=start.cuda(), prefix_len=plen.cuda(), max_prefix_len=P, Kt=Kt, Vt=Vt,
              mask=bits, n_nodes=torch.full((B,), M, dtype=torch.int32, device="cuda"), O=O, lse=lse, workspace=ws, block_table=table, page_size=page)
    assert rb.radar_tree_attention_path(**kw) == (rb.RADAR_ATTN_PATH_FMA if B * Hq * (P + 64) * d <= 294912 else rb.RADAR_ATTN_PATH_TENSOR_CORE)
    rb.radar_tree_attention(ctx, **kw)
    ctx.check_device_status()
    err = rounding = 0.0
    for b in range(B):
        s0, n = int(start[b]), int(plen[b])
        K, V = torch.cat([Kc[s0:s0 + n], Kt[b, :M]]).double(), torch.cat([Vc[s0:s0 + n], Vt[b, :M]]).double()
        for h in range(Hq):
            sc = Q[b, :M, h].double() @ K[:, h * Hkv // Hq].T * d ** -0.5
            sc[:, n:] = sc[:, n:].masked_fill(~low[b, :M, :M], float("-inf"))
            ref = sc.softmax(-1) @ V[:, h * Hkv // Hq]
            err += float((O[b, :M, h].double() - ref).square().sum())
            rounding += float((ref.to(torch.bfloat16).double() - ref).square().sum())
            assert float((lse[b, h, :M].double() - sc.logsumexp(-1)).abs().max()) < 4e-6
    assert err ** 0.5 <= 1.001 * rounding ** 0.5
    ctx.close()


@pytest.mark.parametrize("Hq,Hkv,d", [(129, 1, 64), (260, 2, 128)])
def test_ratios_above_128_run_on_the_fma_kernel(Hq, Hkv, d):
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx, B, P, M = rb.Context(0), 2, 300, 40
    g = torch.Generator(device="cuda").manual_seed(Hq)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    Q, Kt, Vt, Kc, Vc = rand(B, 64, Hq, d), rand(B, 64, Hkv, d), rand(B, 64, Hkv, d), rand(B * P, Hkv, d), rand(B * P, Hkv, d)
    O = torch.zeros_like(Q)
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.RADAR_BF16, P), dtype=torch.uint8, device="cuda")
    bits = ((torch.ones(64, dtype=torch.int64) << torch.arange(1, 65)) - 1).cuda().repeat(B, 1)          # a chain: rows 0 .. i
    kw = dict(B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, kv_start=torch.tensor([0, P], device="cuda"), max_prefix_len=P, Kt=Kt, Vt=Vt, mask=bits,
              prefix_len=torch.full((B,), P, dtype=torch.int32, device="cuda"), n_nodes=torch.full((B,), M, dtype=torch.int32, device="cuda"),
              O=O, workspace=ws)
    assert rb.radar_tree_attention_path(**kw) == rb.RADAR_ATTN_PATH_FMA
    rb.radar_tree_attention(ctx, **kw)
    ctx.check_device_status()
    for b in range(B):
        K, V = (torch.cat([c[b * P:(b + 1) * P], t[b, :M]]).double().repeat_interleave(Hq // Hkv, 1) for c, t in ((Kc, Kt), (Vc, Vt)))
        sc = torch.einsum("mhd,khd->hmk", Q[b, :M].double(), K) * d ** -0.5
        sc[:, :, P:] = sc[:, :, P:].masked_fill(torch.ones(M, M, device="cuda").triu(1).bool(), float("-inf"))
        ref = torch.einsum("hmk,khd->mhd", sc.softmax(-1), V)
        assert float((O[b, :M].double() - ref).abs().max()) < 2.0 ** -8 * float(ref.abs().max())       # half an ulp of bf16, and then some
    ctx.close()
