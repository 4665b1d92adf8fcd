"""Builds in-tree the CUDA library libpp_attn.so (sm_100a only) and the CPython module _pp_torch_*.so
through which the binding makes the calls of a step."""
from __future__ import annotations

import os
import re
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpp_attn.so")
EXT_SOURCE = "pp_torch.cpp"
SOURCES = ["pp_api.cu", "pp_plan.cu", "pp_fwd.cu", "pp_bwd.cu", "pp_rope.cu", "pp_loss.cu", "pp_rows.cu"]
HEADERS = ["pp_internal.h", "pp_dev.cuh", "pp_ptx.cuh", os.path.join("..", "..", "include", "pp_attn.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _outdated(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(os.path.join(CSRC, d)) > t for d in deps)


def needs_build() -> bool:
    return _outdated(LIB, SOURCES + HEADERS)


def ext_module() -> str:
    """Name of the module: it holds the torch version, and its file name Python's ABI tag, so that a
    module built for others is neither loaded nor taken for up to date."""
    import torch
    return "_pp_torch_" + re.sub(r"\W", "_", torch.__version__)


def ext_path() -> str:
    return os.path.join(HERE, ext_module() + sysconfig.get_config_var("EXT_SUFFIX"))


def _start_ext(force: bool):
    """Starts the compiler for the module if it has to be built."""
    if not force and not _outdated(ext_path(), [EXT_SOURCE, HEADERS[-1]]):
        return None
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f"-DPP_MODULE={ext_module()}"]
    cmd += ["-I" + d for d in include] + [os.path.join(CSRC, EXT_SOURCE), "-o", ext_path(),
                                          "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda",
                                          "-ltorch_cpu", "-ltorch_python"]
    return cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def _finish(procs, verbose: bool):
    """Waits for all compilers, also when one has failed."""
    failed = []
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            failed.append(" ".join(cmd))
    if failed:
        raise RuntimeError("compiler failed: " + "; ".join(failed))


def build(force: bool = False, verbose: bool = False) -> str:
    ext = _start_ext(force)
    procs = [ext] if ext else []
    objs = []
    if not force and not needs_build():
        _finish(procs, verbose)
        return LIB
    for s in SOURCES:
        obj = os.path.join(CSRC, s.replace(".cu", ".o"))
        cmd = [_nvcc(), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
               "-Xcompiler", "-fPIC", "-c", os.path.join(CSRC, s), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        cmd[1:1] = os.environ.get("PP_EXTRA_NVCC_FLAGS", "").split()
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    _finish(procs, verbose)
    link = [_nvcc(), "-shared", "-o", LIB] + objs
    subprocess.run(link, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
