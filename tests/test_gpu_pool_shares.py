"""Boundaries of the pooling shares: written bag by bag with the offsets check where there are few bags per share, searched for
otherwise and with malformed offsets.  Bags of very different lengths, empty ones at both ends, more shares than lookups, one
bag over many shares, and bag counts on both sides of the rule, for each of the pooling kernels that take shares.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums)."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import assert_close, binding, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu


def offsets_of(kind, nb, L, rng):
    if kind == "empty ends":
        cuts = np.sort(rng.integers(0, L + 1, nb - 1))
        cuts[: nb // 3], cuts[-(nb // 3):] = 0, L
    elif kind == "one long bag":
        at = nb // 2
        cuts = np.minimum(np.arange(1, nb), L // 10)
        cuts[at:] = np.maximum(L - (nb - 1 - np.arange(at, nb - 1)), cuts[at - 1])
    else:
        cuts = np.sort(rng.integers(0, L + 1, nb - 1))
    return np.concatenate([[0], cuts, [L]]).astype(np.int64)


@pytest.mark.parametrize("d", [(4, 4, 4), (2, 4, 4), (2, 2, 4), (4, 8, 4)])
@pytest.mark.parametrize("kind,B,L", [("empty ends", 900, 20_000), ("one long bag", 1500, 60_000), ("mixed", 1, 777), ("mixed", 5000, 3),
                                      ("mixed", 5000, 1), ("mixed", 7, 100_000), ("mixed", 140_000, 50_000), ("empty ends", 140_000, 300_000)])
def test_out(binding, d, kind, B, L):  # noqa: F811
    spec = TableSpec(N=3000, n=(15, 15, 14), d=d, r=(1, 8, 8, 1), alpha=1.0, core_dist="normal", core_scale=0.3)
    T = 2
    rng = np.random.default_rng(B + L)
    wl = workloads.custom([spec] * T, B, 1, seed=3)
    wl.offsets = offsets_of(kind, T * B, L, rng)
    wl.indices = rng.integers(0, 3000, L).astype(np.int64)
    assert np.all(np.diff(wl.offsets) >= 0)
    emb = binding.from_workload(wl, enable_backward=True)      # (few lookups make no shares on a handle without it)
    ref = oracle.forward_workload(wl, memo=True)
    for _ in range(2):
        out = emb.forward(dev(wl.indices), dev(wl.offsets), B)
        assert emb.status() == 0
        assert_close(out.cpu().numpy(), ref, "out")
        # malformed offsets in between: the boundaries of the next call do not come from these
        bad = wl.offsets.copy()
        bad[T * B // 2] = L + 5
        emb.forward(dev(wl.indices), dev(bad), B)
        assert emb.status() == binding.STATUS_OFFSETS
    assert emb.check_guards() is None
