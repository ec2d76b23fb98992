"""Build of the CUDA library libmcgpu.so (sm_103a only), in-tree.

The translation units are compiled in parallel with nvcc and linked into
``paper_2305_09130_gb300/_lib/libmcgpu.so`` with the CUDA runtime linked
statically.  Rebuilds only when a source or header is newer than the library.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(PKG, "_lib")
LIB = os.path.join(OUT_DIR, "libmcgpu.so")
SOURCES = ["mc_api.cu", "mc_kernels.cu", "mc_explore_cas.cu", "mc_tree.cu", "mc_cfg.cu", "mc_cfg_jobs.cu", "mc_batch.cu", "mc_noalloc.cu", "mc_roofline.cu", "mc_pe.cu"]
HEADERS = [os.path.join(CSRC, "mc_internal.h"), os.path.join(CSRC, "mc_cfg_jobs.h"), os.path.join(CSRC, "mc_cfg_wave.h"), os.path.join(CSRC, "mc_cfg_wave.cuh"), os.path.join(CSRC, "mc_walk.cuh"), os.path.join(CSRC, "mc_walk.h"), os.path.join(CSRC, "mc_tree.h"), os.path.join(CSRC, "mc_pe_ordered.cuh"), os.path.join(CSRC, "mc_device.cuh"), os.path.join(CSRC, "mc_explore.cuh"), os.path.join(CSRC, "mc_host.h"),
           os.path.join(INCLUDE, "mc.h"), os.path.join(INCLUDE, "mc_pe.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(OUT_DIR, exist_ok=True)
    cc = nvcc()
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-pthread", "-I", INCLUDE,
                    "-I", CSRC]
    objs = []

    def compile_one(src):
        obj = os.path.join(OUT_DIR, os.path.splitext(src)[0] + f".{os.getpid()}.o")
        cmd = [cc] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd))
        subprocess.check_call(cmd)
        return obj

    with cf.ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [cc] + ARCH + ["-shared", "-o", tmp] + objs + ["-cudart", "static", "-Xcompiler", "-pthread"]
    if verbose:
        print(" ".join(cmd))
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    for o in objs:
        os.remove(o)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
