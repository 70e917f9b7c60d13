"""Grouping with the prefix levels scanned in one cluster and links, list and schedule over all SMs, against the integer oracle: on
both sides of its dispatch, units of equal counts and of equal costs, three and four cores, a row buffer too small for all lookups."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, check_grouping, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

EQUAL = ((4, 4, 4), (1, 8, 8, 1))
COSTS = {3: ((3, 3, 5), (1, 6, 4, 1)), 4: ((2, 2, 2, 4), (1, 3, 4, 5, 1))}


# tables, rows, row factors, (dims, ranks), lookups per table, kernel launches of grouping and schedule (least, most)
@pytest.mark.parametrize("T,N,n,shape,L,least,most", [
    (12, 400_000, (74, 74, 74), EQUAL, 2731, 6, 6),          # 6 k words: from 2^15 lookups on
    (12, 400_000, (74, 74, 74), EQUAL, 2730, 4, 4),
    (12, 400_000, (74, 74, 74), COSTS[3], 2731, 4, 4),       # equal costs: not where the cluster takes all steps
    (33, 100_000, (47, 47, 47), EQUAL, 3, 6, 6),             # past the words of the cluster's other steps
    (33, 100_000, (47, 47, 47), COSTS[3], 60, 9, 9),
    (9, 16_000_000, (64, 64, 64, 64), COSTS[4], 999, 9, 9),
    (38, 16_000_000, (256, 256, 250), EQUAL, 70, 6, 6),      # 97 k words and past the limit
    (39, 16_000_000, (256, 256, 250), EQUAL, 70, 12, 20),
])
def test_grouping_and_rows(binding, T, N, n, shape, L, least, most):  # noqa: F811
    d, r = shape
    spec = TableSpec(N=N, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3)
    rng = np.random.default_rng(T + L)
    B = max(1, L // 7)
    wl = workloads.custom([spec] * T, B, 1, seed=L)
    emb = None
    for rep in range(2):
        rows = np.concatenate([np.minimum(rng.integers(0, N, L), rng.integers(0, N, L)) if rep else rng.integers(0, N, L) for _ in range(T)])
        rows[:2] = 0, N - 1
        cuts = np.sort(rng.integers(0, L + 1, (T, B - 1)), axis=1) + L * np.arange(T)[:, None]
        wl.indices = rows.astype(np.int64)
        wl.offsets = np.concatenate([np.concatenate([[t * L], cuts[t]]) for t in range(T)] + [[T * L]]).astype(np.int64)
        if emb is None:
            emb = binding.from_workload(wl, enable_backward=True)
        binding.launch_count(reset=True)
        out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
        took = binding.launch_count() - 2 - (emb.K == 4)      # a sweep kernel, the pooling, the level-2 products
        assert least <= took <= most, took
        assert emb.status() == 0
        check_grouping(emb, wl)
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")
    assert emb.check_guards() is None


def test_more_lookups_than_rows_fit(binding):  # noqa: F811
    # a list without room for all marked prefixes is not made from the marks: the call goes the way it went, and reports
    spec = TableSpec(N=100_000, n=(47, 47, 47), d=EQUAL[0], r=EQUAL[1], alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec] * 33, 60, 1, seed=3)
    for room, status in ((wl.L, 0), (wl.L // 2, binding.STATUS_OVERFLOW)):
        emb = binding.from_workload(wl, enable_backward=True, max_unique_rows=room)
        binding.launch_count(reset=True)
        emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
        took = binding.launch_count() - 2
        assert (took == 6) == (room == wl.L), took
        assert emb.status() & binding.STATUS_OVERFLOW == status
        assert emb.check_guards() is None
