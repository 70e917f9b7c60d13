"""Backward sweeps that stream the rows of a batch of groups (ranks 8 and 16 with C of 16, 8 and 4 rows, rank 32 with C of 4 rows):
groups of 1 to 5 rows (a step holds four), around 32 rows (a block of steps, where sums of dC are handed over) and of several
hundred rows, in ranks that are no multiple of eight before them, three and four cores (the left operand through the parent),
rows and prefixes dropped at the row capacity; rebuilt products of rank 8 and gradients of short groups as exact as without the stream.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums, 3xTF32 products)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), (8, 8)), ((2, 4, 4), (5, 8)), ((4, 4, 4), (16, 16)), ((4, 4, 4), (5, 16)), ((2, 4, 4), (16, 16)), ((2, 4, 4), (3, 16)), ((2, 2, 4), (32, 32)), ((2, 2, 4), (16, 16))]


def ids_with_groups(n, sizes, rng):
    """Row ids whose length-2 prefixes hold sizes[i % len] rows each."""
    rows = []
    for i, p in enumerate(rng.permutation(n[0] * n[1])):
        rows.append(p * n[2] + rng.choice(n[2], min(sizes[i % len(sizes)], n[2]), replace=False))
    return np.concatenate(rows)


@pytest.mark.parametrize("d,r", SHAPES)
@pytest.mark.parametrize("n,sizes", [((3, 7, 9), (1, 2, 3, 4, 5)), ((2, 9, 140), (31, 32, 33, 1, 35, 64, 128, 140)), ((1, 1, 700), (700,)), ((37, 5, 6), (1, 6))])
def test_gradients(binding, d, r, n, sizes):  # noqa: F811
    spec = TableSpec(N=int(np.prod(n)), n=n, d=d, r=(1,) + r + (1,), alpha=1.0, core_dist="normal", core_scale=0.3)
    rng = np.random.default_rng(len(sizes) + n[2])
    T, B = 2, 50
    wl = workloads.custom([spec] * T, B, 1, seed=1, with_grad=True)
    per_table = [np.concatenate([x, rng.choice(x, 40)]) for x in (ids_with_groups(n, sizes, rng) for _ in range(T))]
    per_table = [rng.permutation(x) for x in per_table]
    wl.indices = np.concatenate(per_table).astype(np.int64)
    cuts, at = [], 0
    for x in per_table:
        cuts += [at + c for c in [0] + sorted(rng.integers(0, len(x) + 1, B - 1).tolist())]
        at += len(x)
    wl.offsets = np.array(cuts + [at], dtype=np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) >= 0
    ref = oracle.backward_workload(wl)
    for rep in range(2):
        out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
        emb.backward(dev(wl.grad_out))
        grads = emb.get_grads()
        for t in range(T):
            for k in range(3):
                assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.status() == 0 and emb.check_guards() is None


@pytest.mark.parametrize("d,r", SHAPES)
@pytest.mark.parametrize("n,cap", [((6, 8, 40), 301), ((30, 32, 2), 77)])     # fewer groups than rows kept; more
def test_rows_dropped_at_the_capacity(binding, d, r, n, cap):  # noqa: F811
    # the last groups keep some or none of their rows; what is left is the gradient of the rows that were kept
    spec = TableSpec(N=1920, n=n, d=d, r=(1,) + r + (1,), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], 60, 12, seed=4, with_grad=True)
    rng = np.random.default_rng(2)
    wl.indices = rng.integers(0, 1920, wl.L).astype(np.int64)
    kept = np.unique(wl.indices)[:cap]
    emb = binding.from_workload(wl, enable_backward=True, max_unique_rows=cap)
    emb.forward(dev(wl.indices), dev(wl.offsets), 60)
    assert emb.status() == binding.STATUS_OVERFLOW
    emb.backward(dev(wl.grad_out))
    grads = emb.get_grads()
    keep = np.isin(wl.indices, kept)
    wl.offsets = np.concatenate([[0], np.cumsum(keep)])[wl.offsets].astype(np.int64)
    wl.indices = wl.indices[keep]
    ref = oracle.backward_workload(wl)
    for k in range(3):
        assert_close(grads[0][k], ref[0][k], f"dG[0][{k}]")
    assert emb.check_guards() is None


@pytest.mark.parametrize("ra,b", [(8, 1), (8, 4), (5, 4), (16, 12), (7, 2), (32, 31)])
def test_rebuilt_products_of_rank_8_in_fp32(binding, ra, b):  # noqa: F811
    # C = x * 1 + 1 * (-1) with x = 1 + 2^-11 + 2^-23: both products and their sum are exact in fp32, while an operand split into two
    # TF32 values has lost the last bit of x, 2^-12 of C.  Everything after C is exact: dG_K = 16 C * lookups of the row.
    x = 1.0 + 2.0 ** -11 + 2.0 ** -23
    spec = TableSpec(N=60, n=(3, 4, 5), d=(4, 4, 4), r=(1, ra, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], 40, 3, seed=ra, with_grad=True)
    g0, g1, g2 = (np.zeros_like(c) for c in wl.cores[0])
    g0[0, :, :, 0], g0[0, :, :, b] = 1.0, 1.0
    g1[0], g1[b] = x, -1.0
    g2[:] = 1.0
    wl.cores = [[g0, g1, g2]]
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == 2
    emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    emb.backward(dev(np.ones((wl.B, 64), dtype=np.float32)))
    got = emb.get_grads()[0][2].astype(np.float64)
    lookups = np.bincount(wl.indices % 5, minlength=5)
    ref = np.broadcast_to((16.0 * (x - 1.0) * lookups)[None, :, None, None], got.shape)
    assert np.max(np.abs(got - ref)) <= 2.0 ** -21 * np.max(ref)   # sums of at most 120 exact terms of 13 bits


@pytest.mark.parametrize("d,r", [s for s in SHAPES if s != ((2, 4, 4), (5, 8))])   # (8 x 8 is left to fp32 multiply-adds)
@pytest.mark.parametrize("rows", [1, 2, 5])
def test_gradient_of_a_product_in_one_sum_per_pair_of_rows(binding, d, r, rows):  # noqa: F811
    # A row's part of dC is 1 + 2^-24 + 2^-24 + 0: one sum of four terms gives 1 + 2^-23 (the tensor core keeps bits below the last one
    # until it truncates the result), two terms and then two give 1.  Rows of zeros beside it must not split it.
    n = (1, 1, 8)
    spec = TableSpec(N=8, n=n, d=d, r=(1,) + r + (1,), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], rows, 1, seed=1, with_grad=True)
    wl.indices = np.arange(rows, dtype=np.int64)
    g = [np.zeros_like(c) for c in wl.cores[0]]
    g[0][0, 0, 0, 0] = 1.0                                  # P_1: one row, one column
    g[2][:, rows - 1, :, 0] = [1.0, 2.0 ** -24, 2.0 ** -24, 0.0]
    wl.cores = [g]
    emb = binding.from_workload(wl, enable_backward=True)
    emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    emb.backward(dev(np.ones((wl.B, int(np.prod(d))), dtype=np.float32)))
    got = emb.get_grads()[0][1][0, 0].astype(np.float64)    # [d_2, r_2]: dC of the first row of P_1
    assert np.all(got == 1.0 + 2.0 ** -23)


@pytest.mark.parametrize("d,r,variant", [((2, 2, 4, 4), (5, 16, 16), 1), ((2, 2, 4, 4), (3, 8, 8), 2), ((1, 4, 4, 4), (4, 5, 16), 1), ((1, 4, 4, 4), (3, 7, 8), 2),
                                         ((2, 1, 4, 4), (3, 16, 16), 6), ((2, 1, 2, 4), (4, 32, 32), 8), ((2, 1, 2, 4), (4, 16, 16), 9)])
@pytest.mark.parametrize("n,sizes", [((3, 2, 7, 9), (1, 2, 3, 4, 5)), ((2, 2, 5, 140), (31, 32, 33, 1, 34, 64, 128, 140)), ((7, 5, 5, 6), (1, 6, 2))])
def test_four_cores(binding, d, r, variant, n, sizes):  # noqa: F811
    spec = TableSpec(N=int(np.prod(n)), n=n, d=d, r=(1,) + r + (1,), alpha=1.0, core_dist="normal", core_scale=0.3)
    rng = np.random.default_rng(len(sizes) + n[3])
    T, B = 2, 50
    wl = workloads.custom([spec] * T, B, 1, seed=1, with_grad=True)
    per_table = [ids_with_groups((n[0] * n[1], n[2], n[3]), sizes, rng) for _ in range(T)]
    per_table = [rng.permutation(np.concatenate([x, rng.choice(x, 40)])) for x in per_table]
    wl.indices = np.concatenate(per_table).astype(np.int64)
    starts = np.concatenate([[0], np.cumsum([len(x) for x in per_table])])
    cuts = [np.sort(rng.integers(a, b + 1, B - 1)) for a, b in zip(starts, starts[1:])]
    wl.offsets = np.concatenate([np.concatenate([[a], c]) for a, c in zip(starts, cuts)] + [starts[-1:]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == variant
    out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for t in range(T):
        for k in range(4):
            assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.status() == 0 and emb.check_guards() is None


@pytest.mark.parametrize("d,r", [((4, 4, 4), (16, 16)), ((2, 2, 4), (32, 32)), ((4, 8, 4), (32, 32)), ((3, 4, 5), (4, 3))])   # units of equal group counts; the last by cost
@pytest.mark.parametrize("L", [700, 40_000])     # one cluster; marks of the digit-major order beside the row scan
def test_prefixes_dropped_at_the_capacity(binding, d, r, L):  # noqa: F811
    # 900 prefixes and more in a batch with room for 77 nodes: the marks made from all prefixes are made again from those that are kept
    spec = TableSpec(N=1920, n=(30, 32, 2), d=d, r=(1,) + r + (1,), alpha=1.0, core_dist="normal", core_scale=0.3)
    B, cap = 60, 77
    wl = workloads.custom([spec], B, 1, seed=4, with_grad=True)
    rng = np.random.default_rng(L)
    wl.indices = rng.integers(0, 1920, L).astype(np.int64)
    wl.offsets = np.concatenate([[0], np.sort(rng.integers(0, L + 1, B - 1)), [L]]).astype(np.int64)
    kept = np.unique(wl.indices)[:cap]
    emb = binding.from_workload(wl, enable_backward=True, max_unique_rows=cap)
    emb.forward(dev(wl.indices), dev(wl.offsets), B)
    assert emb.status() == binding.STATUS_OVERFLOW
    emb.backward(dev(wl.grad_out))
    grads = emb.get_grads()
    keep = np.isin(wl.indices, kept)
    wl.offsets = np.concatenate([[0], np.cumsum(keep)])[wl.offsets].astype(np.int64)
    wl.indices = wl.indices[keep]
    ref = oracle.backward_workload(wl)
    for k in range(3):
        assert_close(grads[0][k], ref[0][k], f"dG[0][{k}]")
    assert emb.check_guards() is None
