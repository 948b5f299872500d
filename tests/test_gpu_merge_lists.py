"""The merge of a row's chunk lists at the counts where its bound changes (one list, fewer lists than k, 32 and more; small and
large chunks): top-k and log-probability of radar_expand_step against torch, with the best values spread out, all in one list, and
equal across lists (lower token first).  Tolerance: 16 ulp of the fp32 sums of a chunk plus the rounding of the logits' sum."""
import pytest

from paper_2512_14069_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,V", [(2, 4091), (2, 8190), (2, 36000), (2, 126976), (2, 131072), (2, 131077), (40, 60000), (40, 73728)])
@pytest.mark.parametrize("k", [1, 10, 32])
def test_merge_of_lists(B, V, k):
    import torch
    from paper_2512_14069_b200 import binding as rb
    from paper_2512_14069_b200.pipeline import SpecStep
    ctx = rb.Context(0)
    g = torch.Generator(device="cuda").manual_seed(V + k)
    s = SpecStep(ctx, B=B, V=V, k=k, t_max=1, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16)
    gate = {n: torch.from_numpy(x).cuda() for n, x in W.gate_weights(W.shrink(W.CONFIGS[2], k=k, t_max=2)).items()}
    for best in ("spread", "one list", "equal"):
        logits = torch.randn(B, 1, V, device="cuda", generator=g)
        if best == "one list":
            logits[:, :, 100:100 + k] += 20
        elif best == "equal":
            logits[:, :, 17::(V - 17) // 40] = 9.0
        ref = logits[:, 0].double()
        order = torch.sort(ref, dim=-1, descending=True, stable=True).indices[:, :k]
        lp = torch.log_softmax(ref, -1).gather(1, order)
        for pipelined in (True, False):
            s.run_expansion(logits, gate, pipelined=pipelined)
            ctx.check_device_status()
            assert torch.equal(s.topk_tok1[:, 0].long(), order)
            assert float((s.topk_logp1[:, 0].double() - lp).abs().max()) < 2e-6 + 32 * 2 ** -24
    ctx.close()
