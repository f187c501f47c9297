"""In-tree build of the CUDA library: nvcc for sm_100a -> libkvp.so next to this file; and of the binding's argument
packing: g++ against torch's headers -> _pack.so.

Run as ``python -m paper_2608_15943_b200.build`` or call ``build()``.  Objects are rebuilt only
when a source or header is newer than the object; _pack.so also when it was built for another Python or torch.
"""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
HEADER = os.path.join(os.path.dirname(HERE), "include", "kvp.h")
LIB = os.path.join(HERE, "libkvp.so")
PACK = os.path.join(HERE, "_pack.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

SOURCES = ["kvp_common.cu", "kvp_plan.cu", "kvp_gemm.cu", "kvp_attn_fwd.cu", "kvp_attn_bwd.cu", "kvp_decode.cu", "kvp_misc.cu", "kvp_stage.cu",
           "kvp_api.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
         "--expt-relaxed-constexpr", "-Xptxas", "-v"] + os.environ.get("KVP_NVCC_EXTRA", "").split()


def _newest_header() -> float:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    hs.append(HEADER)
    return max(os.path.getmtime(h) for h in hs)


def _compile(src: str, force: bool) -> str:
    obj = os.path.join(OBJ, src.replace(".cu", ".o"))
    path = os.path.join(CSRC, src)
    if not force and os.path.exists(obj) and os.path.getmtime(obj) > max(os.path.getmtime(path), _newest_header()):
        return obj
    cmd = [NVCC, *FLAGS, "-c", path, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    with open(obj + ".log", "w") as fh:
        fh.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    return obj


def _pack_key(torch_dir: str) -> str:
    """What _pack.so is built against: its layout of torch's and Python's objects holds for these alone."""
    with open(os.path.join(torch_dir, "version.py")) as fh:
        return f"{sys.version}\n{torch_dir}\n{fh.read()}"


def _build_pack(force: bool) -> None:
    src = os.path.join(CSRC, "kvp_pack.cpp")
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    key, key_file = _pack_key(torch_dir), os.path.join(OBJ, "_pack.key")
    if not force and os.path.exists(PACK) and os.path.getmtime(PACK) > max(os.path.getmtime(src), os.path.getmtime(HEADER)) and os.path.exists(key_file):
        with open(key_file) as fh:
            if fh.read() == key:
                return
    inc, lib = os.path.join(torch_dir, "include"), os.path.join(torch_dir, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-w", "-I" + sysconfig.get_paths()["include"],
           "-I" + inc, "-I" + os.path.join(inc, "torch", "csrc", "api", "include"), src, "-o", PACK, "-L" + lib,
           "-ltorch_python", "-ltorch_cpu", "-lc10", "-Wl,-rpath," + lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed for {src}:\n{r.stdout}\n{r.stderr}")
    with open(key_file, "w") as fh:
        fh.write(key)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    srcs = [s for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]
    with ThreadPoolExecutor(max_workers=min(8, len(srcs) + 1)) as ex:
        pack = ex.submit(_build_pack, force)
        objs = list(ex.map(lambda s: _compile(s, force), srcs))
        pack.result()
    if force or not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs):
        cmd = [NVCC, "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a", "-lcudart_static",
               "-ldl", "-lpthread", "-lrt"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    if verbose:
        for o in objs:
            with open(o + ".log") as fh:
                sys.stdout.write(fh.read())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
