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
