"""Guard bytes between the counters and the row bitmap, which share one clear: damage there is seen, and a call leaves them as they are."""
import pytest

import workloads
from test_gpu_parity import binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

COUNTERS = 4 * (16 + 64)   # bytes of status word and counters
BITMAP = 512               # from the status word to the row bitmap


@pytest.mark.parametrize("N", [900, 5_000_000])   # one cluster for everything; row scan as kernels of its own
@pytest.mark.parametrize("at", [COUNTERS, COUNTERS + 100, BITMAP - 1])
def test_damage_behind_the_counters(binding, N, at):  # noqa: F811
    n = round(N ** (1 / 3)) + 1
    spec = TableSpec(N=N, n=(n, n, n), d=(4, 4, 4), r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    wl = workloads.custom([spec], 50, 4, seed=1, with_grad=True)
    emb = binding.from_workload(wl, enable_backward=True)
    assert emb.check_guards() is None
    emb.forward(dev(wl.indices), dev(wl.offsets), wl.B)
    emb.backward(dev(wl.grad_out))
    assert emb.check_guards() is None
    base = (-emb.workspace.data_ptr()) % 256
    found = []
    for block in range(0, 16384, 256):     # regions start on multiples of 256 bytes; behind three small ones comes the status
        byte = emb.workspace[base + block + at:base + block + at + 1]
        before = byte.clone()
        byte += 1
        if emb.check_guards() == "status":
            found.append(block)
        byte.copy_(before)
    assert len(found) == 1
    assert emb.check_guards() is None
