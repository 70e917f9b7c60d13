"""Arithmetic of stacked rows (csrc/rows.cuh), compiled for the host: positions and counts around 2^31 and 2^32 rows, up to
2^31 - 1 nodes of 1024 rows; CTAs per slice for 2^31 slices and more."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_03459_b200", "csrc")
SOURCE = """
#include "rows.cuh"
extern "C" {
uint64_t rows(uint32_t nodes, int M) { return tt_stacked_rows(nodes, M); }
uint64_t at(uint64_t row, int M) { StackedRow r = tt_stacked_row(row, M); return ((uint64_t)r.node << 32) | r.m; }
uint64_t after(uint32_t node, uint32_t m, uint32_t n, int M) { StackedRow r = {node, m}; r = tt_stacked_next(r, n, M); return ((uint64_t)r.node << 32) | r.m; }
int ctas(int sm_count, int64_t slices, int64_t tiles) { return tt_ctas_per_slice(sm_count, slices, tiles); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    where = tmp_path_factory.mktemp("rows")
    (where / "rows.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(where / "rows.so"), str(where / "rows.cpp")], check=True)
    so = ctypes.CDLL(str(where / "rows.so"))
    so.rows.restype = so.at.restype = so.after.restype = ctypes.c_uint64
    so.rows.argtypes = [ctypes.c_uint32, ctypes.c_int]
    so.at.argtypes = [ctypes.c_uint64, ctypes.c_int]
    so.after.argtypes = [ctypes.c_uint32] * 3 + [ctypes.c_int]
    so.ctas.argtypes = [ctypes.c_int, ctypes.c_int64, ctypes.c_int64]
    return so


@pytest.mark.parametrize("nodes,M", [(1, 1), (33_554_432, 64), (16_777_216, 256), (67_108_864, 64), (4_300_000, 1000), (2**31 - 1, 1024)])
def test_positions(lib, nodes, M):
    total = nodes * M
    assert lib.rows(nodes, M) == total
    for row in {0, 1, M - 1, M, total // 2, 2**31 - 1, 2**31, 2**32 - 64, 2**32 + 63, total - 65, total - 1}:
        if not 0 <= row < total:
            continue
        assert lib.at(row, M) == (row // M) << 32 | row % M
        for n in (0, 1, 31, 32, 63, 64):
            if row + n < total:
                assert lib.after(row // M, row % M, n, M) == ((row + n) // M) << 32 | (row + n) % M


@pytest.mark.parametrize("slices,tiles,want", [
    (1, 1, 1), (1, 10**12, 2368), (60, 1, 1), (60, 100, 40), (2368, 9, 1), (3 * 800_000_000, 1, 1), (2**31 - 1, 2**40, 1), (2**40, 5, 1)])
def test_ctas_per_slice(lib, slices, tiles, want):
    assert lib.ctas(148, slices, tiles) == want
