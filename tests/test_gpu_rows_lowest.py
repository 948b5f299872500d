"""Log-probabilities of rows with masked tokens at large negative values, the type's lowest among them, where whole runs of tokens
are masked (a padded vocabulary, a few allowed tokens), and of rows with large logits: a span of such values must not spoil the
row's normaliser.  Few rows (a cluster to each) and many (pass and merge kernels); against fp64."""
import pytest

from test_gpu_expand_calls import ctx       # noqa: F401  (a fixture)
from test_gpu_rows_masked import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [1000, 9001, 131072])
@pytest.mark.parametrize("low", [-1e5, -1e9, -1e10, -3e20, -1e38, None])        # None: the type's lowest value
@pytest.mark.parametrize("copies", [1, 43])          # 43 * 7 rows: more than a cluster each
def test_runs_of_masked_tokens(ctx, dtype, V, low, copies):     # noqa: F811
    import torch
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    low = torch.finfo(dt).min if low is None else low
    g = torch.Generator(device="cuda").manual_seed(V)
    x = torch.randn(7, V, device="cuda", generator=g) * 3
    x[1, V - V // 3:] = low                          # the end of the vocabulary
    x[2, 40:] = low                                  # its beginning is allowed,
    x[3, :V - 20] = low                              # ... its end
    keep = torch.randperm(V, device="cuda", generator=g)[:30]
    x[4] = torch.full_like(x[4], low).scatter(0, keep, x[4][keep])
    x[5, V // 4: V // 2] = low
    x[6, ::2] = low
    _check(ctx, x.to(dt), 10, copies)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [1000, 9001, 131072])
def test_rows_at_large_values(ctx, dtype, V):     # noqa: F811
    """Rows that lie at a large value as a whole: their log-probabilities are those of the same row at zero, to the fp64 sums'
    rounding."""
    import torch
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    x = torch.zeros(6, V, device="cuda")
    for r, at in enumerate([-1e9, 1e9, 1e7, -1e7, 2.0 ** 17, -(2.0 ** 17)]):
        x[r] = at
    _check(ctx, x.to(dt), 10, 1)
