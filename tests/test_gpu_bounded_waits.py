"""The bounded waits of the tensor-core attention: long enough for any healthy kernel, and bounded."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def waits(tmp_path_factory):
    from paper_2512_14069_b200 import build
    so = str(tmp_path_factory.mktemp("waits") / "libwaits.so")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *build.FLAGS, "-shared", "-I" + build.CSRC,
                           os.path.join(HERE, "bounded_waits.cu"), "-o", so])
    return ctypes.CDLL(so)


def test_a_wait_gives_up_after_seconds(waits):
    """A wait for an arrival that never comes returns false, after more than a second (a healthy launch can be held up for tens
    of milliseconds, by the memory system or by its neighbours) and less than a minute; those behind it cost microseconds."""
    import torch
    ns, seen = torch.zeros(3, dtype=torch.int64, device="cuda"), torch.ones(3, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert waits.waits_that_run_out(ctypes.c_void_p(ns.data_ptr()), ctypes.c_void_p(seen.data_ptr())) == 0
    assert not seen.any()
    took = ns.tolist()
    assert all(1e9 < t < 6e10 for t in took[:2]), took
    assert took[2] < 1e8, took
