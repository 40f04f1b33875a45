"""Builds libmgdense.so (sm_100a only) next to this file with nvcc, and the native views (_mgviews.*.so), the part of the binding that makes
torch tensors, with g++; no JIT cache is used."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmgdense.so")
OBJ_DIR = os.path.join(HERE, "build")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def views_path() -> str:
    """The native views lay torch's and Python's structures out as their headers have them: a file of its own for each pair of versions."""
    import torch
    return os.path.join(HERE, f"_mgviews.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so")


def _views_command(src: str):
    import torch
    from torch.utils import cpp_extension
    includes = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], *cpp_extension.include_paths()]
    libs = cpp_extension.library_paths()
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *[f for d in includes for f in ("-isystem", d)], src, "-o", views_path(), *[f"-L{d}" for d in libs], "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10"]


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    extra_flags = tuple(extra_flags) + tuple(os.environ.get("MG_NVCC_FLAGS", "").split())
    os.makedirs(OBJ_DIR, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers += [os.path.join(ROOT, "include", f) for f in os.listdir(os.path.join(ROOT, "include"))]
    nvcc = _nvcc()
    objs, jobs = [], []
    for src in sources():
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            jobs.append([nvcc, *NVCC_FLAGS, *extra_flags, "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0 or verbose:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("compiler failed: " + " ".join(cmd))

    # (the library does without the views, so it is there whatever becomes of them, and the views need what the library does not: Python's headers)
    views_src, views = os.path.join(CSRC, "mg_views.cpp"), None
    with ThreadPoolExecutor(max_workers=max(1, min(8, len(jobs) + 1))) as ex:
        if force or _stale(views_path(), [views_src, os.path.join(ROOT, "include", "mgdense.h")]):
            if os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h")):
                views = ex.submit(run, _views_command(views_src))
            else:
                sys.stderr.write("no Python.h: the native views are left out, and views of an export take longer\n")
        list(ex.map(run, jobs))
        if jobs or force or _stale(LIB, objs):
            run([nvcc, "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a",
                 "-Xcompiler", "-fPIC", "-lcudart_static", "-ldl", "-lpthread", "-lrt"])
    if views:
        views.result()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
