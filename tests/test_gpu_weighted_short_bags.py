"""Weighted and mean pooling of short bags (windows across bags): one-lookup bags, windows with one boundary, with many, with
bags that span sub-warps and windows, with empty bags and with ids outside the table, both staged row widths.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [(4, 4, 4), (2, 4, 4), (2, 3, 4)])
@pytest.mark.parametrize("bags", [(1, 1), (1, 3), (5, 9), (2, 20), (0, 3), (31, 33), (0, 40)])
def test_out_and_gradients(binding, d, bags):  # noqa: F811
    spec = TableSpec(N=500, n=(7, 8, 9), d=d, r=(1, 8, 8, 1), alpha=0.7, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec, spec], 701, bags, seed=bags[0] * 100 + bags[1], with_grad=True)
    rng = np.random.default_rng(1)
    weights = rng.standard_normal(wl.L).astype(np.float32)
    for bad in (False, True):
        if bad:
            wl.indices = wl.indices.copy()
            wl.indices[rng.integers(0, wl.L, max(1, wl.L // 50))] = 500
        emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
        for mode, wt in (("mean", None), ("sum", weights)):
            emb.set_pooling(mode, None if wt is None else dev(wt))
            out = emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
            assert_close(out.cpu().numpy(), oracle.forward_workload(wl, weights=wt, mode=mode), f"out {mode} bad={bad}")
            emb.backward(dev(wl.grad_out))
            grads, ref = emb.get_grads(), oracle.backward_workload(wl, weights=wt, mode=mode)
            for t in range(wl.T):
                for k in range(3):
                    assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}] {mode} bad={bad}")
        assert emb.check_guards() is None
