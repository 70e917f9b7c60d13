"""Four-core training calls: the middle levels of shapes that fill the 32 x 32 quarters of their tiles, that do not, and of both in one
handle; with level 2's digit-major list made on a side stream and in line, and as the first call of a handle inside a graph.

Bar: max|err| <= 1e-5 * max|ref| per tensor, the bound of the other parity tests."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

WHOLE32 = ((4, 5, 4, 6), (1, 2, 2, 4), (1, 32, 32, 32, 1))
WHOLE96 = ((3, 4, 3, 5), (2, 1, 2, 4), (1, 64, 96, 32, 1))     # a tile and a half high
RAGGED = ((5, 3, 4, 3), (2, 4, 2, 1), (1, 40, 32, 33, 1))


@pytest.mark.parametrize("shapes,lookups", [([WHOLE32], (0, 90)), ([WHOLE96], (0, 12)), ([WHOLE96], 1), ([RAGGED], (0, 40)), ([WHOLE32, RAGGED], (0, 40))])
def test_four_core_step(binding, shapes, lookups):  # noqa: F811
    import torch
    specs = [TableSpec(N=int(np.prod(n)) - 1, n=n, d=d, r=r, alpha=0.9, core_dist="normal", core_scale=0.2) for n, d, r in shapes]
    wl = workloads.custom(specs, 53, lookups, seed=len(shapes) + shapes[0][2][2], with_grad=True)
    ref = oracle.backward_workload(wl)
    ids, off, grad = dev(wl.indices), dev(wl.offsets), dev(wl.grad_out)

    def check(emb, what):
        grads = emb.get_grads()
        for t in range(wl.T):
            for k in range(4):
                assert_close(grads[t][k], ref[t][k], f"dG[{t}][{k}] {what}")
        assert emb.check_guards() is None and emb.status() == 0

    emb = binding.from_workload(wl, enable_backward=True)
    out = torch.empty((wl.B, wl.T * wl.D), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        emb.forward(ids, off, wl.B, out)
        emb.backward(grad)
    graph.replay()
    torch.cuda.synchronize()
    check(emb, "first call, captured")
    for serial in (False, True):
        emb = binding.from_workload(wl, enable_backward=True)
        if serial:
            emb.enable_timing(2)
        for _ in range(2):
            emb.forward(ids, off, wl.B)
            emb.backward(grad)
        check(emb, f"serial={serial}")
    # bound to the library's own workspace, which makes no streams, and then the backward, which needs one
    emb = binding.TTEmbeddingBag([s.N for s in specs], [s.n for s in specs], [s.d for s in specs], [s.r for s in specs], wl.B, wl.L, enable_backward=True)
    if emb.workspace_bytes <= binding.lib.tt_emb_static_workspace_limit():
        bound = binding.from_workload(wl, enable_backward=True)
        emb.cores, emb.grads = bound.cores, bound.grads
        emb.forward_static(ids, off, wl.B)
        emb.backward(grad)
        check(emb, "static")
