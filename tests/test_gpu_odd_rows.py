"""Rows whose length is no multiple of four floats (staged as the 16-byte pieces that they touch) in the pooling and in the row
gradients, at the lengths where the number of pieces and the kernel change, with `out` and `grad_out` that start off a 16-byte
boundary, weights, mean, bad ids and empty bags; rows of 128 floats in the row gradients.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums)."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


def shifted(x, by):
    """A copy of x that starts `by` floats past an aligned address."""
    flat = torch.empty(x.numel() + by, dtype=torch.float32, device="cuda")[by:]
    return flat.view(x.shape).copy_(x)


@pytest.mark.parametrize("d", [(3, 1, 1), (1, 2, 5), (1, 1, 29), (2, 3, 5), (3, 3, 5), (1, 1, 61), (1, 2, 31), (3, 7, 5), (4, 4, 4), (2, 2, 4), (4, 8, 4)])
@pytest.mark.parametrize("mode", ["sum", "weighted", "mean"])
def test_out_and_gradients(binding, d, mode):  # noqa: F811
    spec = TableSpec(N=230, n=(5, 6, 8), d=d, r=(1, 4, 3, 1), alpha=0.8, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec, spec, spec], 61, (0, 80), seed=sum(d), with_grad=True)
    rng = np.random.default_rng(3)
    wl.indices = wl.indices.copy()
    wl.indices[rng.integers(0, wl.L, wl.L // 40)] = 230
    weights = rng.standard_normal(wl.L).astype(np.float32) if mode == "weighted" else None
    emb = binding.from_workload(wl, enable_backward=True, enable_weighted=True)
    emb.set_pooling("mean" if mode == "mean" else "sum", None if weights is None else dev(weights))
    kw = dict(weights=weights, mode="mean" if mode == "mean" else "sum")
    ref, ref_g = oracle.forward_workload(wl, **kw), oracle.backward_workload(wl, **kw)
    for by in (0, 1, 2):
        out = shifted(torch.zeros(ref.shape, device="cuda"), by)
        emb.forward(dev(wl.indices), dev(wl.offsets), wl.B, out=out)
        assert_close(out.cpu().numpy(), ref, f"out shifted by {by}")
        emb.backward(shifted(dev(wl.grad_out), by))
        grads = emb.get_grads()
        for t in range(wl.T):
            for k in range(3):
                assert_close(grads[t][k], ref_g[t][k], f"dG[{t}][{k}] shifted by {by}")
    assert emb.check_guards() is None


@pytest.mark.parametrize("D,rows", [(45, 1), (61, 2), (3, 5)])
def test_few_rows(binding, D, rows):  # noqa: F811
    # the last row's last piece reaches past the row buffer and past grad_out
    spec = TableSpec(N=rows, n=(1, 1, rows), d=(1, 1, D), r=(1, 2, 2, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], 1, rows, seed=D, with_grad=True)
    wl.indices = np.arange(rows, dtype=np.int64)
    emb = binding.from_workload(wl, enable_backward=True)
    out = emb.forward(dev(wl.indices), dev(wl.offsets), 1)
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
    emb.backward(dev(wl.grad_out))
    grads, ref = emb.get_grads(), oracle.backward_workload(wl)
    for k in range(3):
        assert_close(grads[0][k], ref[0][k], f"dG[{k}]")
    assert emb.check_guards() is None
