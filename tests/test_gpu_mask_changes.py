"""RADAR_EXPAND_VOCAB reads its mask without owning it: a sequence may be stopped, by another stream, while its rows are read.
The pass of the other sequences must not notice, nor any block wait for one that has left: no timeout on the status word, and the
calls that follow give what they give undisturbed.  Sizes: clusters of one, two and eight blocks a row, and the two-kernel form."""
import pytest

from paper_2512_14069_b200 import workloads as W
from test_gpu_expand_calls import ctx       # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,V,k", [(2, 9000, 10), (2, 30000, 10), (2, 128256, 10), (8, 128256, 10)])
def test_mask_changes_while_rows_are_read(ctx, B, V, k):     # noqa: F811
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    t_max = 4
    g = torch.Generator(device="cuda").manual_seed(V)
    draft = torch.randn(B, 1 + (t_max - 1) * k, V, device="cuda", generator=g) * 3
    gate = {n: torch.from_numpy(x).cuda() for n, x in W.gate_weights(W.shrink(W.CONFIGS[2], k=k, t_max=t_max)).items()}
    force = torch.full((B,), t_max, dtype=torch.int32, device="cuda")
    new = lambda: SpecStep(ctx, B=B, V=V, k=k, t_max=t_max, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
    ref, s = new(), new()
    for t in (1, 2, 3):
        ref.expand(t, draft, gate, force)
    for t in (1, 2):
        s.expand(t, draft, gate, force)
    mask = torch.ones(B, dtype=torch.uint8, device="cuda")
    flips = torch.cuda.Stream()
    flips.wait_stream(torch.cuda.current_stream())
    for _ in range(200):
        with torch.cuda.stream(flips):
            mask[:1].fill_(0)
            mask[:1].fill_(1)
        s.expand(3, draft, gate, force, phase=rb.RADAR_EXPAND_VOCAB, vocab_mask=mask)
    s.expand(3, draft, gate, force, phase=rb.RADAR_EXPAND_SELECT)
    torch.cuda.synchronize()
    ctx.check_device_status()
    for n in ("frontier_tok", "frontier_score", "topk_tok", "topk_logp", "gate_logits"):
        assert torch.equal(getattr(s, n)[2, 1:], getattr(ref, n)[2, 1:]), n
    s2 = new()
    for t in (1, 2):
        s2.expand(t, draft, gate, force)
    mask.zero_()                                         # nothing is read for a mask of zeros; a mask of ones reads all rows
    s2.expand(3, draft, gate, force, phase=rb.RADAR_EXPAND_VOCAB, vocab_mask=mask)
    mask.fill_(1)
    s2.expand(3, draft, gate, force, phase=rb.RADAR_EXPAND_VOCAB, vocab_mask=mask)
    s2.expand(3, draft, gate, force, phase=rb.RADAR_EXPAND_SELECT)
    ctx.check_device_status()
    for n in ("frontier_tok", "frontier_score", "topk_tok", "topk_logp", "gate_logits", "h", "c"):
        x, y = getattr(s2, n), getattr(ref, n)
        assert torch.equal(x, y) if n in ("h", "c") else torch.equal(x[2], y[2]), n
