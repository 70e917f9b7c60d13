"""Sort of the lookups by row and the walk over the sorted positions: row counts on both sides of a tile of the segment starts (4096),
rows looked up once, a few times and mostly one row, tables that end inside a batch of 32 positions, for each way the row gradients are
summed; with weights and with mean pooling.  Malformed offsets leave rows without lookups: nothing is written out of place.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (two-level fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), (1, 8, 8, 1)), ((2, 2, 4), (1, 8, 16, 1)), ((4, 8, 4), (1, 8, 8, 1)), ((2, 3, 4), (1, 4, 4, 1)), ((3, 3, 5), (1, 3, 2, 1)),
          ((4, 6, 6), (1, 3, 4, 1)), ((2, 2, 2), (1, 3, 2, 1))]


@pytest.mark.parametrize("d,r", SHAPES)
@pytest.mark.parametrize("U,kind", [(1, "once"), (4095, "once"), (4096, "once"), (4097, "few"), (8192, "few"), (5000, "hot")])
def test_gradients(binding, d, r, U, kind):  # noqa: F811
    rng = np.random.default_rng(U + d[1])
    T, B, n = 3, 37, (20, 20, 21)
    specs = [TableSpec(N=8400 - t, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.3) for t in range(T)]
    wl = workloads.custom(specs, B, 1, seed=U, with_grad=True)
    per_table = []
    for t in range(T):                     # U distinct rows in the first table, U / 3 and one in the others
        rows = rng.permutation(8400 - t)[: (U, max(1, U // 3), 1)[t]]
        extra = {"once": rows[:0], "few": rng.choice(rows, 2 * len(rows)), "hot": np.concatenate([np.full(20_000, rows[0]), rng.choice(rows, 500)])}[kind]
        per_table.append(rng.permutation(np.concatenate([rows, extra])))
    lens = [len(x) for x in per_table]
    base = np.concatenate([[0], np.cumsum(lens)])
    wl.indices = np.concatenate(per_table).astype(np.int64)
    cuts = [np.sort(rng.integers(0, lens[t] + 1, B - 1)) + base[t] for t in range(T)]
    wl.offsets = np.concatenate([np.concatenate([[base[t]], cuts[t]]) for t in range(T)] + [[base[T]]]).astype(np.int64)
    weights = rng.random(wl.L).astype(np.float32) + 0.5
    emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
    for mode, wt in (("sum", None), ("sum", weights), ("mean", None)):
        emb.set_pooling(mode, None if wt is None else dev(wt))
        emb.forward(dev(wl.indices), dev(wl.offsets), B)
        emb.backward(dev(wl.grad_out))
        grads, ref = emb.get_grads(), oracle.backward_workload(wl, weights=wt, mode=mode)
        for t in range(T):
            for k in range(3):
                assert_close(grads[t][k], ref[t][k], f"{mode} dG[{t}][{k}]")
    assert emb.check_guards() is None and emb.status() == 0
    # offsets that leave half of the lookups out, then the good ones again
    bad = wl.offsets.copy()
    bad[T * B // 2:] = bad[T * B // 2]
    emb.set_pooling("sum")
    emb.forward(dev(wl.indices), dev(bad), B)
    assert emb.status() & binding.STATUS_OFFSETS
    emb.backward(dev(wl.grad_out))
    assert emb.check_guards() is None
    emb.forward(dev(wl.indices), dev(wl.offsets), B)
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    assert_close(grads[0][2], ref[0][2], "after malformed offsets")
