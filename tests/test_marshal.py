"""The native argument marshaller: every field of every argument struct lands where ctypes puts it, and what does not fit
is refused.  No GPU needed (the called function is a Python callback)."""
import ctypes

import pytest
import torch

from paper_2512_14069_b200 import binding as rb
from paper_2512_14069_b200 import build as rbuild


@pytest.fixture(scope="module", autouse=True)
def built():
    rbuild.build()


def _filler(struct, optional=(), like=None, addresses=True):
    from paper_2512_14069_b200 import _marshal
    kinds = {ctypes.c_int: 0, ctypes.c_int64: 1, ctypes.c_size_t: 1, ctypes.c_float: 2, ctypes.c_void_p: 3}
    return _marshal.Filler(ctypes.sizeof(struct), [(f, getattr(struct, f).offset, kinds[t], like, f not in optional, addresses) for f, t in struct._fields_])


@pytest.mark.parametrize("struct", [rb.ExpandArgs, rb.TreeArgs, rb.AttnArgs, rb.AcceptArgs])
def test_fields_land_where_ctypes_puts_them(struct):
    seen = []

    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    def callee(ctx, args, stream):
        seen.append((ctx, ctypes.string_at(args, ctypes.sizeof(struct)), stream))
        return -3

    values, want = {}, struct()
    for i, (f, t) in enumerate(struct._fields_):
        v = {ctypes.c_int: -7 - i, ctypes.c_float: 0.5 * i}.get(t, (1 << 40) + i)
        values[f] = v
        setattr(want, f, v)
    assert _filler(struct)(ctypes.cast(callee, ctypes.c_void_p).value, 11, 13, values) == -3
    assert seen == [(11, bytes(want), 13)]


def test_what_does_not_fit_is_refused():
    fill = _filler(rb.TreeArgs, optional=("n_keep",), like=torch.zeros(0))
    good = {f: 1 for f, _ in rb.TreeArgs._fields_}
    with pytest.raises(TypeError, match="unexpected keyword argument 'extra'"):
        fill(1, 0, 0, dict(good, extra=1))
    with pytest.raises(TypeError, match="missing required keyword argument 'root_tok'"):
        fill(1, 0, 0, {f: v for f, v in good.items() if f not in ("root_tok", "n_keep")})
    with pytest.raises(OverflowError):
        fill(1, 0, 0, dict(good, B=1 << 31))
    with pytest.raises(ValueError, match="contiguous CUDA tensor"):
        fill(1, 0, 0, dict(good, pool_tok=torch.zeros(3)))
    with pytest.raises(TypeError):
        fill(1, 0, 0, dict(good, pool_tok="x"))


def test_a_number_is_no_tensor():
    """Only fields that are declared to take an address do; for the public calls that is the logits' own offset."""
    fill = _filler(rb.TreeArgs, addresses=False)
    numbers = {f: 1 if t is ctypes.c_int else None for f, t in rb.TreeArgs._fields_}
    for name in ("pool_tok", "tree_mask", "n_keep"):
        for value in (0, 4096, True):
            with pytest.raises(TypeError, match="%s: expected a tensor or None, got" % name):
                fill(1, 0, 0, dict(numbers, **{name: value}))
    for call in (rb._expand, rb._expand_calls, rb._tree, rb._attention, rb._accept):
        assert call.addresses <= {"logits"}


def test_public_calls_refuse_numbers():
    class Ctx:
        handle = None
    tree = {f: 1 if t is ctypes.c_int else None for f, t in rb.TreeArgs._fields_}
    stream = type("S", (), {"cuda_stream": 0})()
    with pytest.raises(TypeError, match="retrieve: expected a tensor"):
        rb.radar_rerank_build_tree(Ctx, stream=stream, **dict(tree, retrieve=12345))


def test_a_marshaller_of_another_torch_is_rebuilt_and_not_used(monkeypatch):
    from paper_2512_14069_b200 import _marshal
    assert _marshal.BUILT_FOR == rbuild.marshal_tag() and torch.__version__ in _marshal.BUILT_FOR and rbuild._marshal_is_current()
    rb._check_marshal()
    monkeypatch.setattr(rbuild, "marshal_tag", lambda: "built for torch 0.0, none")
    assert not rbuild._marshal_is_current()
    with pytest.raises(RuntimeError, match="another one .*build it with"):
        rb._check_marshal()


def test_a_missing_marshaller_is_named_when_the_library_is_loaded(monkeypatch):
    import sys
    import paper_2512_14069_b200 as pkg
    monkeypatch.setattr(rb, "_lib", None)
    monkeypatch.delattr(pkg, "_marshal", raising=False)
    monkeypatch.setitem(sys.modules, "paper_2512_14069_b200._marshal", None)
    with pytest.raises(RuntimeError, match="_marshal.so.*build it with"):
        rb.lib()
