"""Build libcacheback.so (the C-ABI of include/cacheback.h) in-tree with nvcc for sm_103a.

    python -m paper_2609_32046_gb300.build [--force]

Each .cu file compiles to an object in parallel under _build/, then nvcc links
the shared library next to this file.  nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(ROOT, "_build")
LIB_NAME = "libcacheback.so"
LIB_PATH = os.path.join(PKG, LIB_NAME)
SOURCES = ["cb_api.cu", "cb_score.cu", "cb_score_tc.cu", "cb_select.cu", "cb_compact.cu", "cb_gather.cu", "cb_rope.cu",
           "cb_depage.cu"]
# files compiled in several parts at the same time: a macro and its values
PARTS = {"cb_score_tc.cu": ("CB_TC_PART", (0, 64, 128))}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                     "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _deps() -> list:
    out = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    out.append(os.path.join(INCLUDE, "cacheback.h"))
    out.append(os.path.abspath(__file__))
    return out


def up_to_date() -> bool:
    if not os.path.exists(LIB_PATH):
        return False
    t = os.path.getmtime(LIB_PATH)
    return all(os.path.getmtime(p) <= t for p in _deps())


def _units() -> list:
    """(source, object name, extra flags) of every compilation."""
    out = []
    for src in SOURCES:
        stem = os.path.splitext(src)[0]
        macro, values = PARTS.get(src, (None, ()))
        out += [(src, "%s_%d" % (stem, v), ["-D%s=%d" % (macro, v)]) for v in values] or [(src, stem, [])]
    return out


def _compile(unit: tuple, verbose: bool) -> str:
    src, stem, flags = unit
    obj = os.path.join(BUILD_DIR, stem + ".o")
    cmd = [nvcc(), *NVCC_FLAGS, *flags, "-c", os.path.join(CSRC, src), "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s%s" % (src, res.stdout, res.stderr))
    if verbose and (res.stdout or res.stderr):
        sys.stderr.write(res.stdout + res.stderr)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    units = _units()
    with cf.ThreadPoolExecutor(max_workers=len(units)) as ex:
        objs = list(ex.map(lambda u: _compile(u, verbose), units))
    tmp = LIB_PATH + ".tmp%d" % os.getpid()
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc link failed:\n%s%s" % (res.stdout, res.stderr))
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB_PATH)
