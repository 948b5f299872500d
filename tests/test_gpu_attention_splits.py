"""Key splits of the fp32 kernel: one tile of keys, one split, a last split of one key, as many splits as there may be, grids of
one block to many an SM; ragged prefixes whose sequences end splits early.  Reference: fp64 softmax in torch.  fp32
products of at most 128 terms and sums over at most 2112 keys, normalised: 1e-5, the contract of the fp32 path."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,P,M", [(1, 4, 4, 64, 0, 3), (1, 4, 4, 64, 128, 17), (1, 4, 2, 128, 129, 64), (2, 4, 4, 64, 1100, 60),
                                            (1, 2, 1, 128, 2048, 33), (1, 16, 16, 128, 500, 60), (3, 32, 8, 64, 200, 50), (6, 16, 2, 128, 97, 20)])
@pytest.mark.parametrize("ragged", [False, True])
def test_key_splits(B, Hq, Hkv, d, P, M, ragged):
    _compare(B, Hq, Hkv, d, [P // (b + 1) if ragged else P for b in range(B)], P, M)


@pytest.mark.parametrize("Hq,Hkv,d,P,plens", [(1, 1, 64, 32768, [32768]), (1, 1, 64, 4096, [4096, 33, 2000]), (1, 1, 128, 8192, [8000]),
                                              (4, 4, 64, 16384, [16384]), (2, 1, 64, 9000, [9000, 0, 1500, 8999]), (8, 8, 64, 8192, [8192])])
def test_more_splits_than_lanes(Hq, Hkv, d, P, plens):
    """Long prefixes of few heads: the combine takes the splits in batches of 32, sequences end in each of them.  The sums are over
    up to 32768 keys, in up to 128 pieces that are summed in fp32 themselves: the same 1e-5."""
    _compare(len(plens), Hq, Hkv, d, plens, P, 60)


def _compare(B, Hq, Hkv, d, plens, P, M):
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx = rb.Context(0)
    g = torch.Generator(device="cuda").manual_seed(B * P + M)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)
    plen = torch.tensor(plens, dtype=torch.int32)
    start = torch.cumsum(plen.long(), 0) - plen
    Q, Kt, Vt = rand(B, 64, Hq, d), rand(B, 64, Hkv, d), rand(B, 64, Hkv, d)
    Kc, Vc = rand(max(int(plen.sum()), 1), Hkv, d), rand(max(int(plen.sum()), 1), Hkv, d)
    low = torch.tril(torch.rand(B, 64, 64, device="cuda", generator=g) < 0.5) | torch.eye(64, device="cuda", dtype=torch.bool)
    low[:, :, 0] = True
    bits = (low.long() << torch.arange(64, device="cuda")).sum(-1)
    O, lse = torch.zeros_like(Q), torch.zeros(B, Hq, 64, device="cuda")
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.RADAR_F32, P) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    rb.radar_tree_attention(ctx, B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, kv_start=start.cuda(), prefix_len=plen.cuda(), max_prefix_len=P,
                            Kt=Kt, Vt=Vt, mask=bits, n_nodes=torch.full((B,), M, dtype=torch.int32, device="cuda"), O=O, lse=lse, workspace=ws)
    ctx.check_device_status()
    for b in range(B):
        s0, n = int(start[b]), int(plen[b])
        K = torch.cat([Kc[s0:s0 + n], Kt[b, :M]]).double().repeat_interleave(Hq // Hkv, 1)
        V = torch.cat([Vc[s0:s0 + n], Vt[b, :M]]).double().repeat_interleave(Hq // Hkv, 1)
        sc = torch.einsum("mhd,khd->hmk", Q[b, :M].double(), K) * d ** -0.5
        sc[:, :, n:] = sc[:, :, n:].masked_fill(~low[b, :M, :M], float("-inf"))
        ref = torch.einsum("hmk,khd->mhd", sc.softmax(-1), V)
        assert float((O[b, :M].double() - ref).abs().max()) < 1e-5
        assert float((lse[b, :, :M].double() - sc.logsumexp(-1)).abs().max()) < 1e-4
    ctx.close()
