"""Sweeps of the 8-row, rank-64 shape (four cores, or three with a first dim factor of 8): groups of one row and of many, fewer
groups than a batch, batches that span several slices of core K-1, ranks r_{K-2} below 64 and no multiple of four.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (3xTF32 products, folded sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,r,B,pool", [
    ((5, 6, 7, 8), (2, 4, 4, 4), (1, 64, 64, 64, 1), 64, (0, 30)),
    ((2, 2, 40, 3), (2, 4, 4, 4), (1, 64, 64, 64, 1), 64, (1, 20)),    # few groups per slice: batches of several slices
    ((9, 9, 1, 70), (2, 4, 4, 4), (1, 7, 61, 64, 1), 50, (1, 90)),     # one slice, odd rank, long groups
    ((3, 50, 90), (8, 4, 4), (1, 36, 64, 1), 100, (1, 50)),
    ((4, 3, 200), (8, 4, 4), (1, 3, 64, 1), 3, (1, 1)),                # three lookups
    ((6, 4, 5, 33), (1, 8, 4, 4), (1, 5, 64, 64, 1), 200, (1, 9)),
])
def test_rows_and_gradients(binding, n, d, r, B, pool):  # noqa: F811
    spec = TableSpec(N=int(np.prod(n)), n=n, d=d, r=r, alpha=0.8, core_dist="normal", core_scale=0.2)
    wl = workloads.custom([spec, spec], B, pool, seed=int(sum(n)) + r[1], with_grad=True)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == 4
    out = emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for t in range(wl.T):
        for k in range(spec.K):
            assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.check_guards() is None and emb.status() == 0
    for ablation in (1, 4):
        study = binding.from_workload(wl, ablation=ablation)
        assert_close(study.forward(dev(wl.indices), dev(wl.offsets), wl.B).cpu().numpy(), oracle.forward_workload(wl), f"out, switch {ablation}")


def test_backward_rebuilds_the_intermediate_product_in_32_bits(binding):  # noqa: F811
    # one row per slice of the last core, gradients of one row of ones: dG_K is then a row of C = P . G_{K-1} as it was formed.
    # Sums of 64 positive products: rounded in fp32 each sum is off by about 2^-24 sqrt(64 / 3) = 2.8e-7 at most; a chain of 24
    # additions into the truncating accumulator is below the exact sum by about as many halves of 2^-24, 7e-7, every time
    n, d, r = (3, 5, 60), (8, 4, 4), (1, 64, 64, 1)
    spec = TableSpec(N=900, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=1.0)
    wl = workloads.custom([spec], 60, 1, seed=3, with_grad=True)
    wl.cores = [[np.abs(c) for c in wl.cores[0]]]
    prefix = np.arange(60) % 15
    wl.indices = (prefix * 60 + np.arange(60)).astype(np.int64)
    wl.offsets = np.arange(61, dtype=np.int64)
    wl.grad_out = np.zeros((60, 128), dtype=np.float32)
    for i in range(60):
        wl.grad_out[i, 4 * (i % 32):4 * (i % 32) + 4] = 1.0
    emb = binding.from_workload(wl, enable_backward=True)
    emb.forward(dev(wl.indices), dev(wl.offsets), 60)
    emb.backward(dev(wl.grad_out))
    got, ref = emb.get_grads()[0][2].astype(np.float64), oracle.backward_workload(wl)[0][2]
    assert np.abs((got - ref) / ref).max() <= 1e-6
    assert abs(((got - ref) / ref).mean()) <= 2e-7
