"""Any-shape backward with a last dim factor below eight that is no multiple of four: every factor, ranks below, at and above four, slices
that are whole float4s and not, rows of C below and above what a thread takes, two to four cores, chunks of many rows and of few; and
what keeps the general items: other last factors beside, rows past the staged ones, few lookups.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests (fp32 sums, eight rows to a partial sum)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes,bags", [
    ([((20, 30, 9), (2, 2, 1), (1, 5, 3, 1))], 420),
    ([((20, 30, 9), (3, 1, 2), (1, 4, 8, 1))], 420),
    ([((12, 10, 60), (2, 3, 3), (1, 6, 6, 1))], 420),
    ([((70, 60, 9), (3, 3, 5), (1, 6, 4, 1))], 420),          # groups of few rows, units of many groups
    ([((20, 30, 40), (1, 1, 5), (1, 2, 9, 1))], 420),
    ([((20, 30, 40), (2, 5, 6), (1, 3, 5, 1))], 420),
    ([((6, 4, 900), (1, 4, 7), (1, 7, 16, 1))], 420),         # groups of hundreds of rows
    ([((3, 5000), (4, 7), (1, 13, 1))], 420),                 # K = 2: units end inside groups
    ([((6, 5, 7, 30), (2, 2, 2, 3), (1, 3, 9, 5, 1))], 420),
    ([((20, 30, 9), (3, 9, 7), (1, 4, 6, 1))], 420),          # D = 189: chunks of fewer rows than threads
    ([((20, 30, 9), (4, 9, 6), (1, 4, 6, 1))], 420),          # D = 216: past the staged rows
    ([((20, 30, 9), (3, 4, 5), (1, 4, 6, 1)), ((9, 30, 9), (5, 4, 3), (1, 4, 6, 1))], 210),   # two last factors
    ([((20, 30, 9), (3, 4, 5), (1, 4, 6, 1)), ((9, 30, 9), (4, 3, 5), (1, 8, 7, 1))], 210),   # one, two shapes
    ([((70, 60, 9), (3, 3, 5), (1, 6, 4, 1))], 20),           # few lookups
])
def test_rows_and_gradients(binding, shapes, bags):  # noqa: F811
    specs = [TableSpec(N=int(np.prod(n)), n=n, d=d, r=r, alpha=0.5, core_dist="normal", core_scale=0.3) for n, d, r in shapes]
    wl = workloads.custom(specs, bags, (0, 90), seed=bags + len(shapes), with_grad=True)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == -1
    out = emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for t in range(wl.T):
        for k in range(specs[0].K):
            assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.check_guards() is None and emb.status() == 0
