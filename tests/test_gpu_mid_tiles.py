"""Middle-core backward of the shapes without a register-tiled kernel (64 x 64 tiles): slices at, below and above one tile,
odd rows and columns, more stacked rows than a pass, slices without nodes, first-core slices that are not 16-byte aligned.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (3xTF32 products, folded sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import TOL, assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,r", [
    ((3, 5, 7), (4, 8, 4), (1, 32, 32, 1)),          # 32 x 256 slices: half a tile high, four wide
    ((6, 4, 5), (2, 4, 2), (1, 64, 16, 1)),          # exactly one tile
    ((40, 3, 6), (2, 5, 2), (1, 65, 13, 1)),         # 65 x 65: a second tile of one row / column, long node lists
    ((2, 9, 4), (1, 1, 3), (1, 1, 1, 1)),            # 1 x 1
    ((7, 6, 5), (3, 3, 5), (1, 6, 4, 1)),
    ((9, 4, 3), (3, 2, 2), (1, 128, 20, 1)),         # two tiles of a
    ((4, 5, 4, 6), (2, 4, 4, 4), (1, 64, 64, 64, 1)),
    ((3, 4, 5, 3), (3, 2, 3, 2), (1, 5, 7, 9, 1)),
    ((3, 9500, 3), (2, 5, 2), (1, 65, 3, 1)),        # so many slices that the CTAs of dG make Y too; two tiles of a
    ((90, 4800, 2), (3, 3, 5), (1, 6, 4, 1)),
])
def test_gradients_and_fused_update(binding, n, d, r):  # noqa: F811
    spec = TableSpec(N=int(np.prod(n)) - 1, n=n, d=d, r=r, alpha=0.9, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec], 37, (0, 40), seed=int(np.prod(d)) + r[1], with_grad=True)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) in (-1, 3, 4)
    for fused in (False, True):
        emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
        emb.backward_sgd(dev(wl.grad_out), 0.01) if fused else emb.backward(dev(wl.grad_out))
        grads, ref = emb.get_grads(), oracle.backward_workload(wl)
        for t in range(wl.T):
            for k in range(spec.K):
                assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}] fused={fused}")
    cores = emb.get_cores()
    for t in range(wl.T):
        for k, want in enumerate(oracle.sgd(wl.cores[t], ref[t], 0.01)):
            assert np.abs(cores[t][k] - want).max() <= TOL * np.abs(want).max()
    assert emb.check_guards() is None and emb.status() == 0
