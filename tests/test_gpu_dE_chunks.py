"""Row-gradient sums (dE) at the borders of a warp's chunk of sorted positions: rows that end on, one before and one after
a border, rows that span a few chunks and rows that span many, vector and scalar row widths, weighted pairs.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (two-level fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [(4, 4, 4), (2, 2, 4), (4, 8, 4), (3, 3, 5), (1, 2, 3), (5, 5, 13), (4, 8, 8)])
@pytest.mark.parametrize("L,hot", [(1, 0.0), (31, 0.9), (33, 0.5), (1000, 0.99), (70_001, 0.5), (300_000, 0.6)])
def test_rows_across_chunk_borders(binding, d, L, hot):  # noqa: F811
    rng = np.random.default_rng(L + d[0])
    n = (4, 5, 6)
    spec = TableSpec(N=120, n=n, d=d, r=(1, 3, 2, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], 16, 1, seed=L, with_grad=True)
    rows = np.where(rng.random(L) < hot, 7, rng.integers(0, 120, L)).astype(np.int64)   # row 7: most of the lookups
    cuts = np.sort(rng.integers(0, L + 1, 15))
    wl.indices, wl.offsets = rows, np.concatenate([[0], cuts, [L]]).astype(np.int64)
    weights = rng.random(L).astype(np.float32)
    emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
    for wt in (None, weights):
        emb.set_pooling("sum", None if wt is None else dev(wt))
        emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
        emb.backward(dev(wl.grad_out))
        grads, ref = emb.get_grads(), oracle.backward_workload(wl, weights=wt)
        for k in range(3):
            assert_close(grads[0][k], ref[0][k], f"dG[{k}]")
    assert emb.check_guards() is None and emb.status() == 0


@pytest.mark.parametrize("d", [(2, 2, 4), (2, 4, 4), (4, 4, 4), (4, 8, 4), (3, 3, 5)])
def test_pieces_around_half_a_chunk_and_blocks_of_32(binding, d):  # noqa: F811
    # chunks of 32 positions (128 and more for rows of 128 floats): rows whose last piece is half a chunk, one more and one less; one piece, a
    # block of 32 pieces, one more, 33 blocks; between rows that shift their first position
    lens = [32 * k + off for k in (1, 2, 31, 32, 33) for off in (-17, -16, -15, -1, 0, 1, 15, 16, 17)] + [32 * 1024 + 5, 32 * 33 * 4, 128 * 32 - 64, 128 * 33 + 65]
    rng = np.random.default_rng(d[1])
    lens = np.concatenate([[x, s] for x, s in zip(rng.permutation(lens), rng.integers(1, 32, len(lens)))])
    L = int(lens.sum())
    assert len(lens) <= 120 and L < 1 << 17
    wl = workloads.custom([TableSpec(N=120, n=(4, 5, 6), d=d, r=(1, 3, 2, 1), alpha=1.0, core_dist="normal", core_scale=0.3)], 16, 1, seed=L, with_grad=True)
    wl.indices = rng.permutation(np.repeat(np.arange(len(lens)), lens)).astype(np.int64)
    wl.offsets = np.concatenate([[0], np.sort(rng.integers(0, L + 1, 15)), [L]]).astype(np.int64)
    weights = rng.random(L).astype(np.float32)
    emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
    for wt in (None, weights):
        emb.set_pooling("sum", None if wt is None else dev(wt))
        for _ in range(3):      # (the warps arrive in another order)
            emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
            emb.backward(dev(wl.grad_out))
            grads, ref = emb.get_grads(), oracle.backward_workload(wl, weights=wt)
            for k in range(3):
                assert_close(grads[0][k], ref[0][k], f"dG[{k}]")
    assert emb.check_guards() is None and emb.status() == 0
