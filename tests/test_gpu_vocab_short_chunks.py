"""Rows whose last chunk is short (a few values to a few warps of vectors, aligned and not): the top-k and the log-normaliser
of radar_expand_step against torch, for fewest and most k.  Values are distinct, so tokens must agree; the log-probability
is an fp32 sum of at most 8192 exponentials a chunk, merged in fp64: 16 ulp of the sum, 2e-6."""
import pytest

from paper_2512_14069_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tail", [1, 7, 31, 33, 250, 256, 260, 1023, 1025, 1030, 1105, 2049])
@pytest.mark.parametrize("k", [1, 10, 32])
def test_short_last_chunk(dtype, tail, k):
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    ctx = rb.Context(0)
    V, B, dt = 4096 + tail, 2, torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(tail * 64 + k)
    if dt == torch.bfloat16:                             # distinct bf16 values: the order of 16-bit patterns of one sign and beyond
        pat = torch.randperm(30000, device="cuda", generator=g)[:B * V]
        logits = ((pat % 15000 + 100).to(torch.int16) | ((pat >= 15000).to(torch.int16) << 15)).view(torch.bfloat16).view(B, 1, V).clone()
        logits = torch.where(logits.float().abs() > 60, (logits.float() * 0).to(dt), logits)
    else:
        logits = torch.randn(B, 1, V, device="cuda", generator=g) * 4
    logits[:, :, V - min(tail, k):] = torch.linspace(61, 70, min(tail, k), device="cuda").to(dt)      # the best sit in the short chunk
    s = SpecStep(ctx, B=B, V=V, k=k, t_max=1, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16, logits_dtype=dt)
    gate = {n: torch.from_numpy(x).cuda() for n, x in W.gate_weights(W.shrink(W.CONFIGS[2], k=k, t_max=2)).items()}
    for pipelined in (True, False):
        s.run_expansion(logits, gate, pipelined=pipelined)
        ctx.check_device_status()
        ref = logits[:, 0].double()
        order = torch.sort(ref, dim=-1, descending=True, stable=True).indices[:, :k]      # equal values: lower token first
        assert torch.equal(s.topk_tok1[:, 0].long(), order)
        lp = torch.log_softmax(ref, -1).gather(1, order)
        assert float((s.topk_logp1[:, 0].double() - lp).abs().max()) < 2e-6 + 70 * 2 ** -24
    ctx.close()
