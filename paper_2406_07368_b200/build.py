"""Builds libla_b200.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and beside it _host.so, the native
side of the Python binding (g++ against torch's headers)."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libla_b200.so")
HOST = os.path.join(PKG, "_host.so")
SOURCES = ["la_api.cu", "decode.cu", "prefill_simt.cu", "prefill_walk.cu", "prefill_tc.cu", "prefill_grouped.cu", "seqpar.cu", "verify.cu", "verify_tc.cu", "commit.cu", "accept.cu", "selftest.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _newer(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(d) <= t for d in deps)


def _built_for(stamp: str, what: str) -> bool:
    """Whether the last build noted in the file `stamp` was made for `what`."""
    if not os.path.exists(stamp):
        return False
    with open(stamp) as f:
        return f.read() == what


def _build_host(deps: list[str]) -> None:
    """_host.so: links against libla_b200.so (found beside it) and the torch libraries of the running interpreter.  Built
    anew for another interpreter or another torch: it uses torch's C++ classes, whose layout changes between versions."""
    import sysconfig
    from importlib.metadata import version

    src, stamp = os.path.join(CSRC, "host.cpp"), os.path.join(OBJ, "host.stamp")
    what = f"python {sysconfig.get_config_var('SOABI')}, torch {version('torch')}"
    if _newer(HOST, [src, *deps]) and _built_for(stamp, what):
        return
    from torch.utils import cpp_extension
    inc = [f"-I{d}" for d in (*cpp_extension.include_paths("cuda"), sysconfig.get_paths()["include"], os.path.join(ROOT, "include"), CSRC)]
    libs = [f"-L{d}" for d in cpp_extension.library_paths("cuda")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", HOST, *inc, *libs, f"-L{PKG}",
           "-lla_b200", "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("g++ failed on host.cpp")
    with open(stamp, "w") as f:
        f.write(what)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "la.h"))
    nvcc = _nvcc()
    flags = list(FLAGS)
    if verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ, src.replace(".cu", ".o"))
        path = os.path.join(CSRC, src)
        if not force and not verbose and _newer(obj, [path] + headers):
            return obj
        cmd = [nvcc, *flags, "-c", path, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        return obj

    with ThreadPoolExecutor(max_workers=min(8, len(SOURCES))) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    if force or not _newer(LIB, objs):
        cmd = [nvcc, "-shared", "-o", LIB, *objs, "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    _build_host([h for h in headers if h.endswith(".h")] + ([LIB] if force else []))
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
