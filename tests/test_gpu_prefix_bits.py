"""Prefix bitmaps written from the bits of the level below, on both sides of the largest radix for which they are (512), with row counts
that end inside a word, a prefix or a digit, beside the row scan and in one cluster, two to four cores; more nodes than there
is room for are in test_gpu_row_stream.py.  Row scan in tiles of 512 words and in longer ones."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, check_grouping, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [
    ((3, 512), 3 * 512), ((40, 512), 40 * 512 - 31), ((40, 513), 40 * 513 - 1),
    ((5, 7, 512), 5 * 7 * 512 - 500), ((5, 513, 31), 5 * 513 * 31 - 32), ((2, 512, 512), 2 * 512 * 512 - 511), ((70, 33, 1), 70 * 33), ((90, 1, 32), 90 * 32 - 3),
    ((3, 4, 5, 33), 3 * 4 * 5 * 33 - 40), ((2, 3, 512, 6), 2 * 3 * 512 * 6 - 1)])
@pytest.mark.parametrize("L", [900, 33_000])      # one cluster; row scan as kernels of its own
def test_grouping(binding, n, N, L):  # noqa: F811
    K = len(n)
    d, r = {2: ((4, 4), (1, 3, 1)), 3: ((4, 4, 4), (1, 8, 8, 1)), 4: ((2, 2, 2, 4), (1, 3, 4, 5, 1))}[K]
    spec = TableSpec(N=N, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3)
    T, B = 3, 64
    rng = np.random.default_rng(N + L)
    wl = workloads.custom([spec] * T, B, 1, seed=L)
    sparse = rng.integers(0, N, 40)
    wl.indices = np.concatenate([rng.integers(0, N, L // 2), rng.choice(sparse, L // 4), np.full(L // 4, N - 1)]).astype(np.int64)
    M = len(wl.indices)
    wl.offsets = np.concatenate([[0], np.sort(rng.integers(0, M + 1, T * B - 1)), [M]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)      # (without it few lookups are not grouped)
    for _ in range(2):
        out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
        assert emb.status() == 0
        check_grouping(emb, wl)
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")
    assert emb.check_guards() is None


@pytest.mark.parametrize("T,N,L", [(1, 131_073, 1 << 18), (1, 131_073, (1 << 18) - 1), (2, 4_000_000, 1 << 18), (3, 4_000_000, 1 << 18), (2, 40_000, 300_000)])
def test_row_scan_tiles(binding, T, N, L):  # noqa: F811
    # tiles of 512 words from 256 k lookups and one lookup per word on: full and empty tiles, tables that end inside one
    n = (round(N ** (1 / 3)) + 1,) * 3
    spec = TableSpec(N=N, n=n, d=(2, 2, 4), r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    B = 500
    rng = np.random.default_rng(T + L)
    wl = workloads.custom([spec] * T, B, 1, seed=L)
    wl.indices = np.where(rng.random(L) < 0.6, rng.integers(0, min(N, 33_000), L), rng.integers(0, N, L)).astype(np.int64)
    wl.indices[:2] = 0, N - 1
    wl.offsets = np.concatenate([[0], np.sort(rng.integers(0, L + 1, T * B - 1)), [L]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)      # (without it few lookups are not grouped)
    out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
    assert emb.status() == 0
    check_grouping(emb, wl)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")
    assert emb.check_guards() is None
