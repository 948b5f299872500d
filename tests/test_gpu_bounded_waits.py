"""The bounded waits of the tensor-core attention: long enough for any healthy kernel, bounded, and for the kernel's own work
only, whatever its predecessor takes."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def waits(tmp_path_factory):
    from paper_2512_14069_b200 import build
    so = str(tmp_path_factory.mktemp("waits") / "libwaits.so")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *build.FLAGS, "-shared", "-I" + build.CSRC,
                           os.path.join(HERE, "bounded_waits.cu"), "-o", so])
    return ctypes.CDLL(so)


def test_the_phase_that_a_block_drains(waits):
    """Every slot of a ring of loads is waited for in the phase it was last armed for (a slot never armed: the one that a new
    barrier passes), after any number of loads.  No GPU needed."""
    for ring in (2, 3):
        for loads in range(5 * ring):
            armed = [len(range(slot, loads, ring)) for slot in range(ring)]
            for slot in range(ring):
                expect = (armed[slot] - 1) & 1
                assert waits.ring_parity(slot, loads % ring, ((loads // ring) & 1) ^ 1) == expect, (ring, loads, slot)


@pytest.mark.gpu
def test_waits_that_run_out(waits):
    """A wait for an arrival that never comes returns false, after more than a second (a healthy launch can be held up for tens
    of milliseconds, by the memory system or by its neighbours) and less than a minute; those behind it cost microseconds.  A
    block's wait for what it has in flight is bounded as well."""
    import torch
    ns, seen = torch.zeros(4, dtype=torch.int64, device="cuda"), torch.ones(4, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert waits.waits_that_run_out(ctypes.c_void_p(ns.data_ptr()), ctypes.c_void_p(seen.data_ptr())) == 0
    assert not seen.any()
    took = ns.tolist()
    assert all(1e9 < t < 6e10 for t in took[:2]), took
    assert took[2] < 1e8, took
    assert 1e8 < took[3] < 1e10, took


@pytest.mark.gpu
@pytest.mark.parametrize("Hq,page", [(16, 0), (32, 16), (12, 0)])
def test_a_slow_predecessor_is_not_a_timeout(waits, Hq, page):
    """The launch begins while its predecessor, which lets it, still runs for longer than the waits of the kernel are bounded by
    (4 s); results are those of a launch with nothing in front, bit for bit.  A ratio of 3 runs the kernel's other form."""
    import torch
    from paper_2512_14069_b200 import binding as rb
    ctx = rb.Context(0)
    B, M, Hkv, d, P = 2, 64, 4, 128, 700
    g = torch.Generator(device="cuda").manual_seed(Hq)
    randn = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()
    rows = B * (-(-P // 16) * 16)
    Kc, Vc, Q, Kt, Vt = randn(rows, Hkv, d), randn(rows, Hkv, d), randn(B, M, Hq, d), randn(B, M, Hkv, d), randn(B, M, Hkv, d)
    ints = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")
    where = dict(kv_start=None, block_table=ints(list(range(rows // 16))).view(B, -1), page_size=page) if page else \
        dict(kv_start=torch.tensor([0, P], device="cuda"))
    mask = torch.full((B, M), -1, dtype=torch.int64, device="cuda")
    ws = torch.zeros(rb.radar_attn_workspace_bytes(ctx, B, Hq, Hkv, d, rb.RADAR_BF16, P), dtype=torch.uint8, device="cuda")
    plen, nodes = ints([P, P - 100]), ints([M, 40])

    def attend():
        O, lse = torch.zeros_like(Q), torch.zeros(B, Hq, M, device="cuda")
        torch.cuda.synchronize()
        return (O, lse), lambda: rb.radar_tree_attention(
            ctx, B=B, Hq=Hq, Hkv=Hkv, d=d, Q=Q, Kc=Kc, Vc=Vc, prefix_len=plen, max_prefix_len=P, Kt=Kt, Vt=Vt, mask=mask, n_nodes=nodes,
            O=O, lse=lse, workspace=ws, **where)

    plain, run = attend()
    run()
    ctx.check_device_status()
    behind, run = attend()
    assert waits.launch_slow_predecessor(ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), ctypes.c_ulonglong(6_000_000_000)) == 0
    run()
    ctx.check_device_status()
    assert plain[0].any() and all(torch.equal(a, b) for a, b in zip(plain, behind))
    ctx.close()
