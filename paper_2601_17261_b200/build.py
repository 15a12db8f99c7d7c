"""Builds libagzo.so (sm_100a) in-tree with nvcc, and the extension module _agzo_calls, the Python entry to its shortest call,
with the C compiler for the interpreter that runs this.  `python -m paper_2601_17261_b200.build`."""
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
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libagzo.so")
CALLS = os.path.join(HERE, "_agzo_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["agzo_api.cu", "agzo_rmw.cu", "agzo_rmw_tc.cu", "agzo_extract.cu", "agzo_panel_qr.cu", "agzo_extract_tc.cu", "agzo_extract_fused.cu", "agzo_extract_split.cu", "agzo_extract_resident.cu", "agzo_static.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the AGZO CUDA library cannot be built")
    return exe


def _stale(out: str, deps) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "agzo.h"))
    nvcc = _nvcc()
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [nvcc, "-c", s, "-o", o] + FLAGS + (["-Xptxas", "-v"] if verbose else [])
            jobs.append(cmd)

    def run(cmd):
        p = subprocess.run(cmd, capture_output=True, text=True)
        if p.returncode != 0:
            raise RuntimeError("compiler failed: %s\n%s\n%s" % (" ".join(cmd), p.stdout, p.stderr))
        return p.stderr

    with ThreadPoolExecutor(max_workers=4) as ex:
        for log in ex.map(run, jobs):
            if verbose and log:
                print(log)
    if jobs or force or _stale(LIB, objs):
        run([nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a",
                                                  "-lcudart"])
    calls = os.path.join(CSRC, "py_calls.c")
    include = sysconfig.get_paths()["include"]
    header = os.path.join(ROOT, "include", "agzo.h")
    if os.path.exists(os.path.join(include, "Python.h")) and (force or _stale(CALLS, [calls, header])):
        run([shutil.which("gcc") or "cc", "-shared", "-fPIC", "-O2", "-I", include, "-I", os.path.dirname(header), calls, "-o", CALLS])
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
