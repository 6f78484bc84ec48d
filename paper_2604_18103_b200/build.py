"""Builds in-tree the C-ABI CUDA library, paper_2604_18103_b200/libdash.so (sm_100a only), and the binding's C part for the running interpreter,
_pycall.<its tag>.so.  The library needs nvcc alone; where the C part cannot be built (no C compiler, no Python.h) the binding goes through ctypes in its place."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdash.so")
PYCALL = os.path.join(HERE, "_pycall" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["api.cu", "hbm_kernels.cu", "attention.cu", "decode_attention.cu", "gemm.cu", "layer_step.cu"]
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC] + os.environ.get("DASH_NVCC_EXTRA", "").split()


def _stale(out: str, deps: list[str]) -> bool:
    return not os.path.exists(out) or any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def build_pycall(force: bool = False) -> str | None:
    """The binding's C part; None (and nothing of an older source left behind) where it cannot be built."""
    src = os.path.join(CSRC, "pycall.c")
    if not force and not _stale(PYCALL, [src]):
        return PYCALL
    cmd = ["gcc", "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], src, "-o", PYCALL, "-lm"]
    try:
        subprocess.check_call(cmd)
    except (OSError, subprocess.CalledProcessError) as e:
        if os.path.exists(PYCALL):
            os.remove(PYCALL)
        print(f"{os.path.basename(PYCALL)} not built ({e}): decoding calls go through ctypes, 2.7 us of the host each slower", file=sys.stderr)
        return None
    return PYCALL


def build(force: bool = False, verbose: bool = False) -> str:
    inc = os.path.join(ROOT, "include")
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "pycall.c"] + [os.path.join(inc, f) for f in os.listdir(inc)]
    if force or _stale(LIB, deps):
        _build_lib(verbose)
    build_pycall(force)
    return LIB


def _build_lib(verbose: bool) -> None:
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    objs, procs = [], []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        cmd = [NVCC, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd)))
        objs.append(obj)
    for src, p in procs:
        if p.wait() != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    link = [NVCC, "-shared", "-o", LIB, *objs]          # the CUDA runtime is linked statically: no library dependency beyond libc / libstdc++
    subprocess.check_call(link)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
