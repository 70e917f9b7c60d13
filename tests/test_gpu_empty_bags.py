"""Pooling windows with empty bags in them: more bags than a window has rows, runs of empty bags longer than a warp, empty bags on both
sides of the end of a table and of a share, an open bag before and after them, for each row width that is pooled in windows across
bags; sums, weights and mean, with the pairs that the backward sorts.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


def lengths(kind, nb, rng):
    if kind == "sparse":        # seven of ten bags empty, the others of one lookup
        return (rng.random(nb) < 0.3).astype(np.int64)
    if kind == "runs":          # runs of 1 to 90 empty bags between bags of 1 to 50
        x = np.zeros(nb, dtype=np.int64)
        at = 0
        while at < nb:
            x[at] = rng.integers(1, 51)
            at += int(rng.integers(1, 91))
        return x
    if kind == "pairs":
        return rng.integers(0, 3, nb)
    return rng.integers(0, 5, nb)


@pytest.mark.parametrize("d", [(4, 4, 4), (2, 4, 4), (3, 4, 4), (2, 3, 4)])
@pytest.mark.parametrize("kind", ["sparse", "runs", "pairs", "few"])
@pytest.mark.parametrize("T,B", [(1, 3000), (3, 1001), (40, 7), (70, 1)])
def test_out_and_gradients(binding, d, kind, T, B):  # noqa: F811
    spec = TableSpec(N=90, n=(4, 5, 5), d=d, r=(1, 8, 8, 1), alpha=0.7, core_dist="normal", core_scale=0.3)
    rng = np.random.default_rng(T * B)
    wl = workloads.custom([spec] * T, B, 1, seed=T, with_grad=True)
    lens = lengths(kind, T * B, rng)
    lens[0] = max(lens[0], 1)
    wl.offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    wl.indices = rng.integers(0, 90, int(lens.sum())).astype(np.int64)
    weights = rng.standard_normal(len(wl.indices)).astype(np.float32)
    emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
    for mode, wt in (("sum", None), ("sum", weights), ("mean", None)):
        emb.set_pooling(mode, None if wt is None else dev(wt))
        out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
        assert emb.status() == 0
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl, weights=wt, mode=mode), f"out {mode}")
        emb.backward(dev(wl.grad_out))
        grads, ref = emb.get_grads(), oracle.backward_workload(wl, weights=wt, mode=mode)
        for t in range(0, T, 9):
            for k in range(3):
                assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}] {mode}")
    assert emb.check_guards() is None


@pytest.mark.parametrize("d,sums", [((4, 4, 4), 2), ((2, 4, 4), 4)])
@pytest.mark.parametrize("weighted", [False, True])
def test_rows_of_a_bag_in_several_partial_sums(binding, d, sums, weighted):  # noqa: F811
    # Bags of 31 rows, the first of 2^24 and the others of 1, between empty ones: a partial sum that holds the first row loses its ones, the
    # other partial sums keep theirs, and the last additions round to multiples of 2.  One chain would lose all thirty.
    spec = TableSpec(N=40, n=(1, 1, 40), d=d, r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    B, T = 30_000, 2          # enough bags that a warp's share holds several
    wl = workloads.custom([spec] * T, B, 1, seed=2)
    g = [np.zeros_like(c) for c in wl.cores[0]]
    g[0][0, :, :, 0], g[1][0, :, :, 0], g[2][0] = 1.0, 1.0, 1.0
    g[2][0, 0] = 2.0 ** 24
    wl.cores = [g] * T
    lens = np.tile([31, 0, 0, 1], T * B // 4)
    wl.offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    wl.indices = np.tile(np.concatenate([np.arange(31), [39]]), T * B // 4).astype(np.int64)
    emb = binding.from_workload(wl, enable_weighted=True)
    emb.set_pooling("sum", dev(np.ones(wl.L, dtype=np.float32)) if weighted else None)
    out = emb.forward(dev(wl.indices), dev(wl.offsets), B).cpu().numpy().astype(np.float64)
    ref = np.tile([2.0 ** 24 + 30, 0.0, 0.0, 1.0], B // 4)[:, None]
    assert emb.status() == 0
    assert np.max(np.abs(out - ref)) <= -(-31 // sums)   # the ones beside the first row (one less than its rows) and half a unit
    assert np.all(out[1::4] == 0.0) and np.all(out[3::4] == 1.0)
