"""Lookups that malformed offsets leave out of every bag: they add nothing to the gradients, whatever the call before left in the workspace,
for each way the offsets are checked (in one cluster, with the marks, in a kernel of its own).

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (two-level fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


def check_gradients(binding, emb, wl, offsets, what):  # noqa: F811
    s = wl.tables[0]
    emb.forward(dev(wl.indices), dev(offsets), wl.B)
    assert emb.status() == (0 if what == "good" else binding.STATUS_OFFSETS)
    emb.backward(dev(wl.grad_out))
    # the lookups that are in bags, as a batch of their own
    bags = [wl.indices[lo:hi] for lo, hi in zip(offsets[:-1], offsets[1:])]
    kept = np.concatenate([[0], np.cumsum([len(b) for b in bags])]).astype(np.int64)
    ref = oracle.backward(s.n, s.d, s.r, s.N, wl.cores[0], np.concatenate(bags), kept, wl.grad_out, memo=True)
    for k, g in enumerate(emb.get_grads()[0]):
        assert_close(g, ref[k], f"{what} dG[{k}]")
    assert emb.check_guards() is None


@pytest.mark.parametrize("L", [3000, 60_000, (1 << 22) + 1])
def test_repeated_rows(binding, L):  # noqa: F811
    # every row is looked up in a bag as well
    spec = TableSpec(N=700, n=(9, 9, 9), d=(2, 2, 4), r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    B = 120
    rng = np.random.default_rng(L)
    wl = workloads.custom([spec], B, 1, seed=3, with_grad=True)
    wl.indices = np.resize(rng.permutation(700), L).astype(np.int64)
    good = np.concatenate([[0], np.sort(rng.integers(0, L + 1, B - 1)), [L]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    check_gradients(binding, emb, wl, good, "good")
    ends = L // 8 + np.sort(rng.integers(0, L // 2, B + 1))
    falls = np.concatenate([[3 * L // 4], np.linspace(L // 4, L // 2, B // 2), np.linspace(L // 9, L // 5, B // 2)])   # two runs of bags
    for what, offsets in (("ends", ends), ("falls", falls)):
        check_gradients(binding, emb, wl, offsets.astype(np.int64), what)
        check_gradients(binding, emb, wl, good, "good")


SHAPES = [((2, 2, 4), (1, 8, 8, 1)), ((4, 4, 4), (1, 8, 16, 1)), ((4, 8, 4), (1, 8, 8, 1)), ((3, 3, 5), (1, 6, 4, 1)), ((2, 3, 4), (1, 4, 4, 1))]


@pytest.mark.parametrize("d,r", SHAPES)
@pytest.mark.parametrize("rows", [0, 9, 5000])
def test_rows_without_a_bag(binding, d, r, rows):  # noqa: F811
    # every other row of 2 x rows in bags, three times each; lookups of all rows in none
    spec = TableSpec(N=10_400, n=(21, 22, 23), d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3)
    B = 50
    rng = np.random.default_rng(rows)
    wl = workloads.custom([spec], B, 1, seed=4, with_grad=True)
    kept = rng.permutation(np.repeat(2 * np.arange(rows) + 1, 3))
    wl.indices = np.concatenate([kept, rng.permutation(10_400)]).astype(np.int64)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, len(kept) + 1, B - 1)), [len(kept)]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    check_gradients(binding, emb, wl, offsets, "kept")


@pytest.mark.parametrize("d,r", SHAPES)
def test_one_row_without_a_bag_in_every_batch(binding, d, r):  # noqa: F811
    # rows looked up once, chunks of several batches of 32 sorted positions, a row without a bag behind another position of each batch
    spec = TableSpec(N=175_000, n=(56, 56, 56), d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3)
    B = 2000
    rng = np.random.default_rng(5)
    wl = workloads.custom([spec], B, 1, seed=5, with_grad=True)
    batches = 5200
    without = np.array([33 * b + b // 2 % 32 + 1 for b in range(batches)])
    kept = rng.permutation(np.setdiff1d(np.arange(33 * batches), without))
    assert len(kept) == 32 * batches and without[-1] < 175_000
    wl.indices = np.concatenate([kept, without]).astype(np.int64)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, len(kept) + 1, B - 1)), [len(kept)]]).astype(np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    check_gradients(binding, emb, wl, offsets, "kept")
