"""Tensor-core attention launches in which a CTA goes through more segments than the ring they are handed on in has entries, of
one to seven tiles each and of up to nineteen (the ends of a segment and its steady state take different paths of the issuing
warp, from four and five full tiles on), for units of one and two row blocks, contiguous and paged; ratios of three run the
kernel's other form, which has neither the ring nor epilogue warps.  Scores of one size, and scores whose maxima jump by more
than the 2^8 from tile to tile behind which an accumulator is rescaled; outputs that start on 32 bytes, and on 16.  Against fp64;
tolerance of the bf16 path (2e-2 max-abs on O and lse: bf16 P and O)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d,page", [(16, 16, 64, 0), (16, 16, 128, 16), (16, 4, 128, 0), (16, 4, 64, 128), (32, 4, 128, 64), (9, 3, 128, 16)])
def test_many_short_segments(Hq, Hkv, d, page):
    rng = np.random.default_rng(Hq * d + page)
    lens = rng.integers(0, 801, 64)
    lens[:10] = (0, 1, 127, 128, 129, 511, 512, 640, 641, 800)
    _check(Hq, Hkv, d, page, rng, lens)


@pytest.mark.parametrize("Hq,Hkv,d,page,o_shift", [(16, 16, 64, 0, 8), (16, 16, 128, 16, 0), (32, 8, 128, 64, 8), (16, 4, 64, 16, 8),
                                                   (64, 8, 128, 0, 8), (24, 8, 64, 128, 8)])
def test_jumping_maxima_in_long_segments(Hq, Hkv, d, page, o_shift):
    rng = np.random.default_rng(Hq + d + page)
    lens = rng.integers(600, 2305, 12)
    lens[:3] = (2304, 2300, 1024)
    _check(Hq, Hkv, d, page, rng, lens, jumps=True, o_shift=o_shift)


def _check(Hq, Hkv, d, page, rng, lens, jumps=False, o_shift=0):
    """o_shift: elements that O starts behind a 32-byte boundary."""
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx = rb.Context(0)
    B, L, M, G, top = len(lens), 4, 64, Hq // Hkv, int(lens.max())
    nodes = rng.integers(1, M + 1, B)
    nodes[:4] = (1, 64, 17, 33)
    g = torch.Generator(device="cuda").manual_seed(d + page)
    randn = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()
    if page:
        pages = -(-lens // page)
        perm = rng.permutation(int(pages.sum()))
        table = np.zeros((B, -(-top // page)), np.int32)
        at = 0
        for b in range(B):
            table[b, :pages[b]] = perm[at:at + pages[b]]
            at += pages[b]
        rows, start, kw = int(pages.sum()) * page, None, dict(block_table=torch.from_numpy(table).cuda(), page_size=page)
        where = [np.array([table[b, i // page] * page + i % page for i in range(lens[b])], np.int64) for b in range(B)]
    else:
        first = np.concatenate([[0], np.cumsum(lens)[:-1]])
        rows, start, kw = int(lens.sum()), torch.from_numpy(first).cuda(), {}
        where = [first[b] + np.arange(lens[b]) for b in range(B)]
    Kc, Vc = randn(L, rows, Hkv, d), randn(L, rows, Hkv, d)
    if jumps:                                  # every fourth tile or so of a sequence has a key that outdoes all before it
        for b in range(B):
            for t in range(0, int(lens[b]), 384):
                Kc[:, int(where[b][t + int(rng.integers(min(384, lens[b] - t)))])] *= 3.0 + t / 128
    Q, Kt, Vt = randn(L, B, M, Hq, d), randn(L, B, M, Hkv, d), randn(L, B, M, Hkv, d)
    anc = np.tril(rng.random((B, M, M)) < 0.4)
    anc[:, np.arange(M), np.arange(M)] = True
    bits = (anc.astype(np.uint64) << np.arange(M, dtype=np.uint64)).sum(-1, dtype=np.uint64).view(np.int64)
    O = torch.zeros(Q.numel() + o_shift, dtype=Q.dtype, device="cuda")[o_shift:].view(Q.shape)
    assert O.data_ptr() % 32 == 2 * o_shift
    lse = torch.zeros(L, B, Hq, M, device="cuda")
    moved = 0                                  # rows and tiles whose maximum is more than 2^8 above all before it
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.RADAR_BF16, top), dtype=torch.uint8, device="cuda")
    rb.radar_tree_attention(ctx, B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, kv_start=start, prefix_len=torch.from_numpy(lens.astype(np.int32)).cuda(),
                            max_prefix_len=top, Kt=Kt, Vt=Vt, mask=torch.from_numpy(bits).cuda(), n_nodes=torch.from_numpy(nodes.astype(np.int32)).cuda(),
                            O=O, lse=lse, workspace=ws, n_layers=L, **kw)
    ctx.check_device_status()
    for b in range(B):
        n, idx = int(nodes[b]), torch.from_numpy(where[b]).cuda()
        K = torch.cat([Kc[:, idx], Kt[:, b, :n]], 1).double().repeat_interleave(G, 2)
        V = torch.cat([Vc[:, idx], Vt[:, b, :n]], 1).double().repeat_interleave(G, 2)
        S = torch.einsum("lmhd,lkhd->lhmk", Q[:, b, :n].double(), K) / d ** 0.5
        keep = torch.cat([torch.ones(n, len(idx), dtype=torch.bool), torch.from_numpy(anc[b, :n, :n])], 1).cuda()
        S = S.masked_fill(~keep, float("-inf"))
        if jumps:
            tops = torch.stack([x.amax(-1) for x in S[..., :lens[b]].split(128, -1)], -1)
            moved += int((tops[..., 1:] - tops[..., :-1].cummax(-1).values > 8 * np.log(2)).sum())
        assert (torch.einsum("lhmk,lkhd->lmhd", S.softmax(-1), V) - O[:, b, :n].double()).abs().max() < 2e-2, b
        assert (S.logsumexp(-1) - lse[:, b, :, :n].double()).abs().max() < 2e-2, b
        assert not O[:, b, n:].any()
    assert not jumps or moved > 1000
    ctx.close()
