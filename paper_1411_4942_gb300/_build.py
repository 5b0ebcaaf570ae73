"""Builds libpathsample.so (the CUDA library behind include/pathsample.h) in
the package directory with nvcc for sm_103a (GB300)."""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_NAME = "libpathsample.so"
LIB_PATH = os.path.join(PKG, LIB_NAME)
SOURCES = ["ps_load.cu", "ps_sort.cu", "ps_prefix.cu", "ps_sample.cu", "ps_batch.cu", "ps_api.cu", "ps_static.cu", "ps_exact.cu", "ps_ingest.cu", "ps_order.cu", "ps_edges.cu", "ps_probe.cu", "ps_readback.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# host FP64 (the estimates and bars) without fused multiply-adds: on Arm the
# compiler would pick them by inlining, and the last bit of a bar with them
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-I", INCLUDE]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    return "nvcc"


def _tag(extra=()) -> str:
    h = hashlib.sha1()
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name), "rb") as f:
            h.update(name.encode() + f.read())
    with open(os.path.join(INCLUDE, "pathsample.h"), "rb") as f:
        h.update(f.read())
    h.update(" ".join(ARCH + NVCC_FLAGS + list(extra)).encode())
    return h.hexdigest()[:16]


def build(force: bool = False, verbose: bool = False, extra_flags=(), out_path: str | None = None) -> str:
    """Compile every translation unit in parallel and link the shared library
    (to out_path when given, e.g. a variant built with extra -D flags)."""
    lib_path = out_path or LIB_PATH
    tag = _tag(extra_flags)
    tag_path = lib_path + ".tag"
    if not force and os.path.exists(lib_path) and os.path.exists(tag_path):
        with open(tag_path) as f:
            if f.read().strip() == tag:
                return lib_path
    obj_dir = os.path.join(PKG, "_build", tag)
    os.makedirs(obj_dir, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(obj_dir, src.replace(".cu", ".o"))
        cmd = [nvcc(), *ARCH, *NVCC_FLAGS, *extra_flags, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
        if verbose and res.stderr:
            print(res.stderr, file=sys.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = lib_path + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{res.stdout}\n{res.stderr}")
    os.replace(tmp, lib_path)
    with open(tag_path, "w") as f:
        f.write(tag)
    return lib_path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
