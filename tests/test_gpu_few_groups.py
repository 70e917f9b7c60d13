"""Sweeps of batches with few groups, whose units are cut finer: every register-tiled and the wide shape, from one group up to just below
and above the limit, with tables of one group beside a large one.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), 32, 0), ((4, 4, 4), 16, 1), ((4, 4, 4), 8, 2), ((4, 8, 4), 32, 3), ((2, 4, 4, 4), 64, 4), ((2, 4, 4), 32, 5),
          ((2, 4, 4), 16, 6), ((2, 4, 4), 8, 7), ((2, 2, 4), 32, 8), ((2, 2, 4), 16, 9), ((2, 2, 4), 8, 10)]


def step(binding, tables, lookups, d, rank, variant):  # noqa: F811
    K = len(d)
    r = (1,) + (rank,) * (K - 1) + (1,)
    scale = 0.3 if K == 3 else 0.1
    specs = [TableSpec(N=int(np.prod(n)), n=n, d=d, r=r, alpha=0.0, core_dist="normal", core_scale=scale) for n in tables]
    wl = workloads.custom(specs, lookups, 1, seed=lookups + variant, with_grad=True)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.table_variant(0) == variant
    out = emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    groups = int(emb.grouping_counts()[:, -2].sum())
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for t in range(wl.T):
        for k in range(K):
            assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}]")
    assert emb.check_guards() is None and emb.status() == 0
    return groups


@pytest.mark.parametrize("d,rank,variant", SHAPES)
@pytest.mark.parametrize("lookups", [1, 5, 300, 2500])     # one group, a part and a bit, some parts, parts of more than four
def test_few_groups(binding, d, rank, variant, lookups):  # noqa: F811
    first = (3,) if len(d) == 4 else ()
    step(binding, [first + (40, 50, 3), (1,) * len(first) + (1, 1, 2)], lookups, d, rank, variant)


@pytest.mark.parametrize("d,rank,variant", [s for s in SHAPES if s[1] <= 16])
@pytest.mark.parametrize("groups", [(67, 70), (73, 74)])   # just below and above the limit of eight per CTA, four CTAs on each of 148 SMs
def test_around_the_limit(binding, d, rank, variant, groups):  # noqa: F811
    total = step(binding, [groups + (2,)], 37_000, d, rank, variant)
    assert 0.95 * groups[0] * groups[1] < total <= groups[0] * groups[1]
