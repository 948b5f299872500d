"""Builds the CUDA library in-tree with nvcc for sm_100a (no JIT cache), and next to it the native argument marshaller
of the binding, which is compiled against torch's headers."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libradar_b200.so")
SOURCES = ["api.cu", "vocab_pass.cu", "row_topk.cu", "expand.cu", "expand_calls.cu", "tree_build.cu", "tree_attention.cu", "tree_attention_tc.cu", "verify_accept.cu", "train.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
         "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
MARSHAL = os.path.join(HERE, "_marshal.so")


def _torch_dir() -> str:
    from importlib.util import find_spec
    return os.path.dirname(find_spec("torch").origin)


def marshal_tag() -> str:
    """What the marshaller is compiled against: it reads tensors by torch's C++ layout and objects by Python's."""
    import re
    import sysconfig
    with open(os.path.join(_torch_dir(), "version.py")) as f:
        version = re.search(r"__version__ = ['\"](.*?)['\"]", f.read()).group(1)
    return "built for torch %s, %s" % (version, sysconfig.get_config_var("SOABI"))


def _marshal_is_current() -> bool:
    if not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < os.path.getmtime(MARSHAL_SRC):
        return False
    with open(MARSHAL, "rb") as f:                   # the module carries its tag as a string
        return marshal_tag().encode() + b"\0" in f.read()


def _start_marshal(force: bool):
    """Starts the compiler for the marshaller if it is out of date; (process, temporary file) or None."""
    if not force and _marshal_is_current():
        return None
    import sysconfig
    tdir = _torch_dir()
    tmp = MARSHAL + ".%d.tmp" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", '-DRADAR_BUILT_FOR="%s"' % marshal_tag(), "-I" + os.path.join(tdir, "include"),
           "-I" + os.path.join(tdir, "include", "torch", "csrc", "api", "include"), "-I" + sysconfig.get_paths()["include"], MARSHAL_SRC,
           "-o", tmp, "-L" + os.path.join(tdir, "lib"), "-lc10", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True), tmp


def _finish_marshal(started):
    if started is None:
        return
    proc, tmp = started
    out, _ = proc.communicate()
    if proc.returncode != 0:
        sys.stderr.write(out)
        raise RuntimeError("g++ failed on marshal.cpp")
    os.replace(tmp, MARSHAL)


def _deps():
    out = [os.path.join(CSRC, s) for s in SOURCES]
    out += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    out.append(os.path.join(os.path.dirname(HERE), "include", "radar.h"))
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu into objects under _build/ and link libradar_b200.so next to this file; build the marshaller."""
    marshal = _start_marshal(force)
    try:
        return _build_library(force, verbose)
    finally:
        _finish_marshal(marshal)


def _build_library(force: bool, verbose: bool) -> str:
    newest = max(os.path.getmtime(p) for p in _deps())
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    procs = []
    objs = []
    for s in SOURCES:
        obj = os.path.join(bdir, s.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc, *FLAGS, "-c", os.path.join(CSRC, s), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((s, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for s, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("[%s]\n%s\n" % (s, out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
