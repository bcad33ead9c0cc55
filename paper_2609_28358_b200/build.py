"""Builds ``libmq.so`` (the C-ABI library) in-tree with nvcc for sm_100a.

    python -m paper_2609_28358_b200.build [--force] [--verbose]

Each ``csrc/*.cu`` is compiled to an object under ``csrc/build/`` (skipped when up to date) and the
objects are linked into ``paper_2609_28358_b200/libmq.so``.  nvcc cross-compiles: no GPU is needed.
``csrc/mq_torch.cpp`` (host code only: the Python binding's marshalling) becomes ``_mq_torch.so`` beside it, linked to
``libmq.so`` and PyTorch's libraries; without PyTorch the library is built alone.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(PKG, "libmq.so")
BINDING = os.path.join(PKG, "_mq_torch.so")
CXX = os.environ.get("CXX", "g++")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC] + os.environ.get("MQ_NVCC_EXTRA", "").split()


def _newest_header() -> float:
    hs = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return max(os.path.getmtime(h) for h in hs)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    hdr = _newest_header()
    jobs, objs = [], []
    for s in srcs:
        o = os.path.join(OBJ, os.path.basename(s)[:-3] + ".o")
        objs.append(o)
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), hdr):
            cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            jobs.append(cmd)
    cmd, binding_obj = _compile_binding(force)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("compilation failed for " + cmd[-3])

    with ThreadPoolExecutor(max_workers=min(9, len(jobs) + 1)) as ex:
        binding = ex.submit(run, cmd) if cmd else None      # its outcome is asked for after the library has been linked
        list(ex.map(run, jobs))
    if jobs or not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        subprocess.check_call([NVCC, "-shared", "-o", tmp] + objs + ["-lcudart"])
        os.replace(tmp, LIB)
    if binding_obj is None:
        sys.stderr.write("PyTorch is not installed: its binding (_mq_torch.so) is not built\n")
        return LIB
    if binding:
        binding.result()
        with open(binding_obj + ".of", "w") as f:
            f.write(_binding_of())
    if not os.path.exists(BINDING) or os.path.getmtime(binding_obj) > os.path.getmtime(BINDING):
        _link_binding(binding_obj)
    return LIB


def _binding_of() -> str:
    """What a compiled binding belongs to, kept beside its object: it works with this build of PyTorch and this Python only."""
    import torch

    return " ".join(str(v) for v in (torch.__version__, torch.version.git_version, os.path.abspath(torch.__file__), sysconfig.get_config_var("SOABI"), CXX))


def _compile_binding(force: bool):
    """(command, object) of the binding's compilation; the command is None when the object is up to date, both without PyTorch."""
    try:
        import torch
    except ImportError:
        return None, None

    src, obj = os.path.join(CSRC, "mq_torch.cpp"), os.path.join(OBJ, "mq_torch.o")
    newest = max(os.path.getmtime(p) for p in (src, os.path.join(ROOT, "include", "mq.h"), os.path.abspath(__file__)))
    made_for = open(obj + ".of").read() if os.path.exists(obj + ".of") else ""
    if not force and os.path.exists(obj) and os.path.getmtime(obj) >= newest and made_for == _binding_of():
        return None, obj
    t = os.path.join(os.path.dirname(os.path.abspath(torch.__file__)), "include")
    cuda = os.path.dirname(os.path.dirname(os.path.abspath(NVCC)))
    return [CXX, "-O2", "-std=c++17", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), "-I", os.path.join(ROOT, "include"),
            "-isystem", t, "-isystem", os.path.join(t, "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
            "-isystem", sysconfig.get_paths()["include"], "-c", src, "-o", obj], obj


def _link_binding(obj: str) -> None:
    import torch

    tmp = BINDING + ".tmp.%d" % os.getpid()
    subprocess.check_call([CXX, "-shared", "-o", tmp, obj, "-L", PKG, "-l:libmq.so", "-L", os.path.join(os.path.dirname(os.path.abspath(torch.__file__)), "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, BINDING)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
