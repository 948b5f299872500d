"""Top-k of rows whose finite logits lie together and within a few ulps of one another, everything else at -inf: the bound of the
merge then comes from one warp's maxima.  Few rows (a cluster to each) and many (pass and merge kernels), rows on and off a
16-byte boundary.  Logits are compared as they are, so the tokens must be those of a stable sort; log-probabilities as in
test_gpu_expand_ranges.py."""
import pytest

from paper_2512_14069_b200 import workloads as W
from test_gpu_expand_calls import ctx       # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def _top_k(ctx, rows, k):     # noqa: F811
    """Tokens and log-probabilities [rows][k] of a first draft call, a row to a sequence."""
    import torch
    from paper_2512_14069_b200.pipeline import SpecStep
    n, V = rows.shape
    s = SpecStep(ctx, B=n, V=V, k=k, t_max=1, N=8, Hq=4, Hkv=4, d=64, kv_dtype=torch.bfloat16, max_prefix_len=16, logits_dtype=rows.dtype)
    gate = {n: torch.from_numpy(x).cuda() for n, x in W.gate_weights(W.shrink(W.CONFIGS[2], k=k, t_max=2)).items()}
    s.run_expansion(rows.view(n, 1, V), gate, pipelined=False)
    ctx.check_device_status()
    return s.topk_tok1[:, 0].long(), s.topk_logp1[:, 0].double()


def _check(ctx, x, k, copies):     # noqa: F811
    import torch
    tok, got = _top_k(ctx, x.repeat(copies, 1), k)
    order = torch.sort(x.double(), dim=-1, descending=True, stable=True).indices[:, :k]
    assert torch.equal(tok, order.repeat(copies, 1))
    lp = torch.log_softmax(x.double(), -1).gather(1, order).repeat(copies, 1)
    assert torch.equal(got == float("-inf"), lp == float("-inf"))
    fin = torch.isfinite(lp)
    assert float((got - lp)[fin].abs().max()) < 2e-6 + 16 * 2 ** -24


@pytest.mark.parametrize("V", [8200, 8203, 16384, 16386, 128256, 170001])
@pytest.mark.parametrize("k", [9, 10, 16, 32])
@pytest.mark.parametrize("copies", [1, 19])          # 19 * 16 rows: more than a cluster each
def test_close_logits_in_one_place(ctx, V, k, copies):     # noqa: F811
    import torch
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = torch.full((16, V), float("-inf"), device="cuda")
    ulps = lambda shape, n: torch.randint(0, n, shape, device="cuda", generator=g)
    near = lambda base, steps: (torch.full(steps.shape, base, device="cuda").view(torch.int32) + steps.int()).view(torch.float32)
    # the first value of each of 32 groups of 32: k - 2 large ones, the next two an ulp apart, the later token the larger
    first = torch.arange(32, device="cuda") * 32
    for r, (lo, hi) in enumerate([(4, 6), (1, 30), (8, 9), (0, 31)]):
        v = torch.full((32,), 0.5, device="cuda")
        others = torch.tensor([i for i in range(32) if i not in (lo, hi)], device="cuda")[:max(k - 2, 0)]
        v[others] = torch.arange(2, 2 + len(others), device="cuda").float()
        v[lo], v[hi] = 1.0, float(near(1.0, torch.ones(1, dtype=torch.int32, device="cuda")))
        x[r, first + 1024 * (r % 2)] = v
    x[4, first] = 1.0
    x[4, 9 * 32] = near(1.0, torch.full((1,), 31, dtype=torch.int32, device="cuda"))
    # 60 allowed tokens of the first 1024; 4096 in a row, one in a hundred raised by a few ulps; all of 1024 within 32 ulps
    for r in range(5, 9):
        at = torch.randperm(1024, device="cuda", generator=g)[:60]
        x[r, at] = near(-6.0, ulps((60,), 40) - 20)
    for r in range(9, 13):
        at = 1024 * (r - 9) + torch.arange(4096, device="cuda")
        x[r, at] = near(7.0, torch.where(ulps((4096,), 100) == 0, ulps((4096,), 30), torch.zeros(4096, dtype=torch.long, device="cuda")))
    for r in range(13, 16):
        at = V - 1024 - 517 * (r - 13) + torch.arange(1024, device="cuda")
        x[r, at] = near(3.0, ulps((1024,), 32))
    _check(ctx, x, k, copies)
