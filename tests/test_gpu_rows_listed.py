"""Rows of which the merge lists most values, because fewer groups than k have any: short rows, and rows masked to a few groups.
They are thinned out by a better bound before they are ranked; lengths around the lines where that begins, where a thread holds
one more of them, and where the row is scanned instead.  Distinct values, values that tie by the dozen, all equal ones, and a few
allowed tokens; few rows (a cluster to each) and many (pass and merge kernels); tokens must be those of a stable sort."""
import pytest

from test_gpu_expand_calls import ctx       # noqa: F401  (a fixture)
from test_gpu_rows_masked import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [127, 129, 136, 256, 264, 520, 992, 1025, 1984, 1991, 2049, 2200])
@pytest.mark.parametrize("k", [10, 16, 32])
@pytest.mark.parametrize("copies", [1, 43])          # 43 * 7 rows: more than a cluster each
def test_listed_values_are_thinned_out(ctx, dtype, V, k, copies):     # noqa: F811
    import torch
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = torch.randn(7, V, device="cuda", generator=g)
    x[1] = torch.randint(0, 12, (V,), device="cuda", generator=g).float()
    x[2] = -3.0
    x[3] = torch.linspace(4.0, -4.0, V, device="cuda")
    x[4] = torch.linspace(-4.0, 4.0, V, device="cuda")
    x[5, V // 3:] = float("-inf")
    x[6, torch.randperm(V, device="cuda", generator=g)[:V // 4]] = float("-inf")
    _check(ctx, x.to(torch.float32 if dtype == "f32" else torch.bfloat16), k, copies)
