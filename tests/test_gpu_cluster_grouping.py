"""Grouping and schedule in one cluster against the integer oracle, on both sides of the sizes where the library switches
between one cluster for everything, a cluster from the prefix levels on, and a kernel per step; repeated calls on one handle
with other batches (the workspace is cleared by the kernel itself)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, check_grouping, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

# row bitmaps of 4096-word tiles (131072 rows each), prefix bitmaps of 512-word tiles.  Last: 2 one cluster for everything, 1
# from the prefix levels on, 0 a kernel per step
CASES = [
    (1, 31, (4, 3, 3), 5, 2),                 # less than a word of rows
    (3, 131072, (32, 64, 64), 300, 2),        # one full tile per table
    (2, 131073, (33, 64, 64), 2000, 2),       # one row more
    (32, 100_000, (47, 47, 47), 200, 2),      # 32 tiles, 16 k words per level: the most words that one cluster takes
    (33, 100_000, (47, 47, 47), 200, 0),      # one table past it
    (11, 400_000, (74, 74, 74), 300, 1),      # 44 tiles, 5.6 k words per level
    (1, 3_900_000, (158, 158, 158), 32_768, 2),
    (1, 3_900_000, (158, 158, 158), 32_769, 1),
    (1, 16_000_000, (256, 250, 250), 5000, 1),
    (2, 16_000_000, (4000, 4000), 3000, 1),   # K = 2
    (1, 16_000_000, (64, 64, 64, 64), 9000, 1),
    (9, 16_000_000, (256, 256, 250), 999, 0),  # prefix bitmaps past the cluster's
]


def mode(binding, emb, *call):  # noqa: F811
    """The way the call's grouping took, by its launches (one, four, or more), and the outputs."""
    binding.launch_count(reset=True)
    out = emb.forward(*call)
    n = binding.launch_count() - 2 - (emb.K == 4)      # a sweep kernel, the pooling, the level-2 products
    return {1: 2, 4: 1}.get(n, 0 if n >= 6 else f"{n} launches"), out


@pytest.mark.parametrize("T,N,n,L,way", CASES)
def test_grouping_and_rows(binding, T, N, n, L, way):  # noqa: F811
    K = len(n)
    d, r = {2: ((4, 4), (1, 3, 1)), 3: ((4, 4, 4), (1, 8, 8, 1)), 4: ((2, 2, 2, 4), (1, 3, 4, 5, 1))}[K]
    spec = TableSpec(N=N, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3)
    rng = np.random.default_rng(T + L)
    B = max(1, L // 7)
    wl = workloads.custom([spec] * T, B, 1, seed=L)
    emb = None
    for rep in range(3):
        rows = np.concatenate([np.minimum(rng.integers(0, N, L), rng.integers(0, N, L)) if rep else rng.integers(0, N, L) for _ in range(T)])
        rows[:2] = 0, N - 1
        cuts = np.sort(rng.integers(0, L + 1, (T, B - 1)), axis=1) + L * np.arange(T)[:, None]
        wl.indices = rows.astype(np.int64)
        wl.offsets = np.concatenate([np.concatenate([[t * L], cuts[t]]) for t in range(T)] + [[T * L]]).astype(np.int64)
        if emb is None:
            emb = binding.from_workload(wl, enable_backward=True)
        took, out = mode(binding, emb, dev(wl.indices), dev(wl.offsets), B)
        assert took == way
        assert emb.status() == 0
        if T <= 3 or rep == 2:
            check_grouping(emb, wl)
            assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")
    assert emb.check_guards() is None


def test_bad_ids_and_offsets_in_the_cluster(binding):  # noqa: F811
    spec = TableSpec(N=1000, n=(10, 10, 10), d=(4, 4, 4), r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec], 8, 3, seed=5)
    emb = binding.from_workload(wl)
    took, good = mode(binding, emb, dev(wl.indices), dev(wl.offsets), 8)
    good = good.cpu().numpy()
    assert took == 2
    bad = wl.indices.copy()
    bad[5], bad[30] = 1000, -1
    emb.forward(dev(bad), dev(wl.offsets), 8)
    assert emb.status() == binding.STATUS_INDEX
    off = wl.offsets.copy()
    off[4] = 1_000_000
    emb.forward(dev(wl.indices), dev(off), 8)
    assert emb.status() == binding.STATUS_OFFSETS
    assert np.array_equal(emb.forward(dev(wl.indices), dev(wl.offsets), 8).cpu().numpy(), good) and emb.status() == 0


def test_schedule_by_cost_in_the_cluster(binding):  # noqa: F811
    # shapes swept by whole CTAs keep units of equal cost: the scan of the costs runs in the cluster
    spec = TableSpec(N=2000, n=(10, 15, 14), d=(3, 3, 5), r=(1, 6, 4, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec], 300, (0, 9), seed=9)
    emb = binding.from_workload(wl, enable_backward=True)
    took, out = mode(binding, emb, dev(wl.indices), dev(wl.offsets), 300)
    assert took == 2
    check_grouping(emb, wl)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")


# tables swept by CTAs (ranks 8 and 12): from the prefix levels on up to 2 M lookups; tables swept by warps: the scans only (six launches)
@pytest.mark.parametrize("T,B,L,rank,way", [(1, 1 << 18, 1000, 8, 2), (1, (1 << 18) + 1, 1000, 8, 1), (20, 64, 1 << 21, 12, 1), (20, 64, (1 << 21) + 1, 12, 0),
                                            (20, 64, 1 << 21, 8, 0)])
def test_many_offsets_and_many_lookups(binding, T, B, L, rank, way):  # noqa: F811
    N, n = (300_000, (67, 67, 67)) if T > 1 else (100_000, (47, 47, 47))      # 10 k words per level; 512
    spec = TableSpec(N=N, n=n, d=(4, 4, 4), r=(1, 8, rank, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec] * T, B, 1, seed=2)
    rng = np.random.default_rng(L)
    wl.indices = rng.integers(0, N, L).astype(np.int64)
    wl.offsets = np.concatenate([[0], np.sort(rng.integers(0, L + 1, T * B - 1)), [L]]).astype(np.int64)
    emb = binding.from_workload(wl)
    took, out = mode(binding, emb, dev(wl.indices), dev(wl.offsets), B)
    assert took == way and emb.status() == 0
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")
    check_grouping(emb, wl)
