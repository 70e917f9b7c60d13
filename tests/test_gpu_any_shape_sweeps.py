"""Sweeps of shapes without a register-tiled variant: groups with one row and with thousands (K = 2: units that start and end
inside a group), odd and even row counts and ranks of C, last dim factors that are and are not multiples of four, slices of
the last core that are not, the largest C, the study switches.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (fp32 sums, eight rows to a partial sum)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,r", [
    ((3, 5000), (8, 8), (1, 24, 1)),            # three groups of thousands of rows
    ((700, 2), (3, 5), (1, 7, 1)),              # many groups of one or two rows
    ((1, 40), (1, 1), (1, 1, 1)),
    ((5, 300), (1, 4), (1, 128, 1)),
    ((4, 90), (32, 3), (1, 127, 1)),            # C of 32 x 127
    ((3, 50), (1024, 1), (1, 4, 1)),            # the largest D and C of 4096 floats
    ((20, 30, 40), (3, 3, 5), (1, 6, 4, 1)),
    ((20, 30, 9), (9, 3, 2), (1, 5, 3, 1)),     # more than eight rows of P
    ((6, 7, 300), (4, 4, 4), (1, 20, 64, 1)),
    ((6, 7, 30), (2, 4, 8), (1, 12, 12, 1)),
    ((6, 5, 7, 30), (2, 2, 2, 3), (1, 3, 9, 5, 1)),
])
def test_rows_and_gradients(binding, n, d, r):  # noqa: F811
    N = int(np.prod(n))
    spec = TableSpec(N=N, n=n, d=d, r=r, alpha=0.7, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec], 211, (0, 60), seed=N + r[1], with_grad=True)
    if wl.D == 1:
        # the first core's gradient is one number, a sum of 6 k terms: with random signs it can cancel to 1/2000 of the sum of
        # their magnitudes (about 1400), where fp32 is only bound to 2^-24 * 1400 = 8e-5; of one sign it is well conditioned
        wl.grad_out = np.abs(wl.grad_out)
        wl.cores = [[np.abs(c) for c in t] for t in wl.cores]
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == -1
    out = emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for t in range(wl.T):
        for k in range(spec.K):
            assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.check_guards() is None and emb.status() == 0
    for ablation in (1, 2, 4):
        study = binding.from_workload(wl, ablation=ablation)
        assert_close(study.forward(dev(wl.indices), dev(wl.offsets), wl.B).cpu().numpy(), oracle.forward_workload(wl), f"out, switch {ablation}")


@pytest.mark.parametrize("n,d,r", [((2, 3, 400), (3, 3, 5), (1, 6, 4, 1)), ((1, 2, 900), (4, 2, 8), (1, 3, 7, 1))])
def test_gradients_above_the_last_core_repeat_bit_for_bit(binding, n, d, r):  # noqa: F811
    # few groups of many rows: a group's rows are cut into parts, which are added in order.  Every row is looked up once, so that
    # the gradients of the rows do not depend on the order of the sorted look-ups
    rng = np.random.default_rng(7)
    N = int(np.prod(n))
    spec = TableSpec(N=N, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=1.0)
    wl = workloads.custom([spec], N, 1, seed=11, with_grad=True)
    wl.indices, wl.offsets = rng.permutation(N).astype(np.int64), np.arange(N + 1, dtype=np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    first = None
    for _ in range(8):
        emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
        emb.backward(dev(wl.grad_out))
        grads = emb.get_grads()[0][:2]
        first = first or grads
        for k in range(2):
            assert np.array_equal(grads[k], first[k]), k
