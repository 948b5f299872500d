"""How a step's draft calls are divided into ranges: they cover the calls once, in order, whatever a call reads."""
import pytest

from paper_2512_14069_b200.pipeline import _ranges


@pytest.mark.parametrize("call_bytes", [1, 24 << 20, (24 << 20) + 1, 48 << 20, (48 << 20) + 1, 1 << 34])
def test_ranges_cover_the_calls(call_bytes):
    for t_max in range(1, 64):
        r = _ranges(t_max, call_bytes)
        assert [t for a, b in r for t in range(a, b + 1)] == list(range(1, t_max + 1))
        assert max(b - a + 1 for a, b in r) <= 8
