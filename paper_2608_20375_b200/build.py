"""Build libgraft.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

Every source becomes an object under _build/ (rebuilt when it or one of its headers is newer) and the objects are
linked into libgraft.so.
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libgraft.so")
GRAFT_H = os.path.join("..", "..", "include", "graft.h")
ALL_HEADERS = ["common.cuh", "internal.h", "edge_score.cuh", "cosine.cuh", "saba.cuh", GRAFT_H]
# source -> headers it depends on
SOURCES = {
    "api.cu": ALL_HEADERS,
    "vocab_pass.cu": ALL_HEADERS + ["umma.cuh", "vocab_common.cuh", "vocab_rows.cuh"],
    "tdes.cu": ALL_HEADERS,
    "tree.cu": ALL_HEADERS,
    "tdes_train.cu": ["common.cuh", "internal.h", GRAFT_H],
    "saba_fit.cu": ["common.cuh", "internal.h", GRAFT_H],
    "tables_mma.cu": ["common.cuh", "internal.h", "umma.cuh", GRAFT_H],
}
# no --use_fast_math: the fp64 pieces (log-sum-exp fold, SABA) and the fp32 divisions must stay IEEE
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _obj(src: str) -> str:
    return os.path.join(OBJ, src.replace(".cu", ".o"))


def needs_build() -> bool:
    for src, hdrs in SOURCES.items():
        if _stale(_obj(src), [os.path.join(CSRC, src)] + [os.path.join(CSRC, h) for h in hdrs]):
            return True
    return _stale(LIB, [_obj(s) for s in SOURCES])


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    inc = ["-I", os.path.join(HERE, "..", "include")]
    cmds = []
    for src, hdrs in SOURCES.items():
        deps = [os.path.join(CSRC, src)] + [os.path.join(CSRC, h) for h in hdrs]
        if not (force or _stale(_obj(src), deps)):
            continue
        cmds.append([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + inc +
                    ["-c", os.path.join(CSRC, src), "-o", _obj(src)])
    procs = [subprocess.Popen(c) for c in cmds]  # the sources compile side by side
    failed = [c for c, pr in zip(cmds, procs) if pr.wait() != 0]
    if failed:
        raise subprocess.CalledProcessError(1, failed[0])
    if force or _stale(LIB, [_obj(s) for s in SOURCES]):
        subprocess.check_call([nvcc, "-shared", "-o", LIB] + [_obj(s) for s in SOURCES] + ["-lcudart"])
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
