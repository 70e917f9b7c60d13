"""Builds libtt_emb.so (sm_100a only) next to this file with nvcc.  Cross-compiles without a GPU."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = [os.path.join(HERE, "csrc", f) for f in ("api.cu", "grouping.cu", "group_cluster.cu", "direct.cu", "forward.cu", "backward.cu", "noalloc.cu", "probe_tcgen05.cu")]
HDR = [os.path.join(HERE, "csrc", f) for f in ("common.cuh", "scan.cuh", "mma.cuh", "quad_mid.cuh", "group.cuh", "generic.cuh", "wide.cuh", "tiles.cuh", "rows.cuh", "stream.cuh")] + [os.path.join(ROOT, "include", "tt_emb.h")]
SO = os.path.join(HERE, "libtt_emb.so")


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def needs_build() -> bool:
    if not os.path.exists(SO):
        return True
    t = os.path.getmtime(SO)
    return any(os.path.getmtime(p) > t for p in SRC + HDR)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return SO
    cmd = [nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(HERE, "csrc"),
           "-o", SO] + SRC
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    return SO


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(SO)
