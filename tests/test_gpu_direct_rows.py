"""Small forward-only calls, whose rows are made lookup by lookup in one kernel: every kind of shape that it takes (three cores with a
kernel of their own, ranks that are no multiple of eight or of four, two and four cores), one to eight warps per bag, more bags than
warps, both id types, pooling modes, bad ids and offsets; against the oracle, against the grouped path (the forward of a handle with the
backward), and the grouping that the inspection calls make afterwards against the integer oracle.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests (fp32 sums)."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_parity import assert_close, binding, check_grouping, dev  # noqa: F401  (binding: fixture)
from workloads import TableSpec

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), (1, 16, 16, 1)), ((4, 4, 4), (1, 32, 8, 1)), ((4, 4, 4), (1, 4, 32, 1)), ((4, 4, 4), (1, 12, 16, 1)), ((4, 8, 4), (1, 32, 32, 1)),
          ((2, 4, 4), (1, 16, 32, 1)), ((2, 4, 4), (1, 8, 16, 1)), ((2, 4, 4), (1, 20, 8, 1)), ((2, 2, 4), (1, 32, 32, 1)), ((2, 2, 4), (1, 8, 16, 1)),
          ((2, 2, 4), (1, 64, 8, 1)),                                     # with a kernel of their own
          ((4, 4, 4), (1, 6, 16, 1)), ((2, 2, 4), (1, 128, 8, 1)), ((4, 6, 4), (1, 16, 24, 1)), ((2, 8, 8), (1, 4, 4, 1)), ((3, 3, 5), (1, 6, 4, 1)),
          ((5, 3, 7), (1, 3, 9, 1)), ((8, 8), (1, 24, 1)), ((3, 5), (1, 7, 1)), ((2, 4, 4, 4), (1, 64, 64, 64, 1)),
          ((2, 2, 4, 4), (1, 8, 16, 16, 1)), ((2, 3, 2, 3), (1, 5, 3, 7, 1))]
ROWS = {2: (45, 41), 3: (11, 13, 14), 4: (6, 5, 9, 7)}


def build(d, r, B, lens, T, seed):
    n = ROWS[len(d)]
    spec = TableSpec(N=int(np.prod(n)) - 3, n=n, d=d, r=r, alpha=1.0, core_dist="normal", core_scale=0.4)
    wl = workloads.custom([spec] * T, B, lens, seed=seed)
    return wl


def launches(binding, emb, *call):  # noqa: F811
    binding.launch_count(reset=True)
    out = emb.forward(*call)
    return binding.launch_count(), out


@pytest.mark.parametrize("d,r", SHAPES)
@pytest.mark.parametrize("B,lens,T", [(64, 1, 1), (70, (0, 3), 2), (64, (0, 40), 1), (90, (3, 9), 2), (1200, (0, 2), 3)])
def test_out_and_grouping(binding, d, r, B, lens, T):  # noqa: F811
    wl = build(d, r, B, lens, T, seed=B)
    emb = binding.from_workload(wl)
    off = dev(wl.offsets)
    n, out = launches(binding, emb, dev(wl.indices), off, B)
    assert n == 1 or (len(d) == 4 and r[1] == 64 and n >= 4)     # rows of rank 64, one by one, take longer than the grouping
    assert emb.status() == 0
    ref = oracle.forward_workload(wl)
    assert_close(out.cpu().numpy(), ref, "out")
    grouped = binding.from_workload(wl, enable_backward=True)
    m, again = launches(binding, grouped, dev(wl.indices), off, B)
    assert m >= 3
    assert_close(out.cpu().numpy(), again.cpu().numpy(), "grouped")
    check_grouping(emb, wl)
    assert emb.status() == 0 and emb.check_guards() is None
    # 32-bit ids, an output that is not 16-byte aligned, and a call after the grouping of the one before was asked for
    room = torch.full((B * T * emb.D + 1,), 7.0, device="cuda")
    emb.forward(dev(wl.indices.astype(np.int32)), off, B, out=room[1:].view(B, T * emb.D))
    assert float(room[0]) == 7.0
    if n == 1:
        assert torch.equal(room[1:].view_as(out), out)
    check_grouping(emb, wl)


@pytest.mark.parametrize("d,r", [SHAPES[0], SHAPES[8], SHAPES[11], SHAPES[15], SHAPES[18]])
@pytest.mark.parametrize("mode", ["mean", "weights"])
def test_pooling_modes(binding, d, r, mode):  # noqa: F811
    wl = build(d, r, 80, (0, 30), 2, seed=4)
    emb = binding.from_workload(wl, enable_weighted=True)
    weights = np.random.default_rng(0).normal(size=wl.L).astype(np.float32) if mode == "weights" else None
    emb.set_pooling("mean" if mode == "mean" else "sum", None if weights is None else dev(weights))
    n, out = launches(binding, emb, dev(wl.indices), dev(wl.offsets), 80)
    assert n == 1 and emb.status() == 0
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl, weights=weights, mode="mean" if mode == "mean" else "sum"), "out")


@pytest.mark.parametrize("B,lens", [(64, 1), (64, (0, 40)), (2000, (0, 3))])
def test_bad_ids_and_offsets(binding, B, lens):  # noqa: F811
    wl = build((4, 4, 4), (1, 8, 8, 1), B, lens, 2, seed=7)
    N = wl.tables[0].N
    emb = binding.from_workload(wl)
    idx, off = dev(wl.indices), dev(wl.offsets)
    good = emb.forward(idx, off, B).clone()
    for bad_id in (N, -1, 1 << 40):
        ids = wl.indices.copy()
        ids[wl.L // 3] = bad_id
        keep = wl.indices
        wl.indices = ids
        n, out = launches(binding, emb, dev(ids), off, B)
        assert n == 1 and emb.status() == binding.STATUS_INDEX
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
        emb.grouping_counts()
        assert emb.status() == binding.STATUS_INDEX
        wl.indices = keep
    for at, value in ((0, 5), (3, 1 << 40), (B // 2, -9), (2 * B, wl.L - 1), (2 * B, wl.L + 1)):
        keep = wl.offsets
        wl.offsets = keep.copy()
        wl.offsets[at] = value
        n, out = launches(binding, emb, idx, dev(wl.offsets), B)
        assert n == 1 and emb.status() == binding.STATUS_OFFSETS
        emb.grouping_counts()
        assert emb.status() == binding.STATUS_OFFSETS
        wl.offsets = keep
        assert torch.equal(emb.forward(idx, off, B), good) and emb.status() == 0
    check_grouping(emb, wl)
    assert emb.check_guards() is None


def test_capacity_and_graph(binding):  # noqa: F811
    wl = build((4, 4, 4), (1, 16, 16, 1), 128, (1, 4), 2, seed=11)
    ref = oracle.forward_workload(wl)
    # a row buffer for fewer rows: the grouped path, which drops the surplus
    small = binding.from_workload(wl, max_unique_rows=50)
    n, _ = launches(binding, small, dev(wl.indices), dev(wl.offsets), 128)
    assert n >= 3 and small.status() == binding.STATUS_OVERFLOW
    # replayed with other contents, and between calls of the same handle; the inspection calls see the replay's lookups
    emb = binding.from_workload(wl)
    idx, off, out = dev(wl.indices), dev(wl.offsets), torch.empty((128, 128), device="cuda")
    graph = emb.capture_forward(idx, off, 128, out)
    other = build((4, 4, 4), (1, 16, 16, 1), 64, 1, 2, seed=12)
    for shift in (0, 5):
        emb.forward(dev(other.indices), dev(other.offsets), 64)
        ids = (wl.indices + shift) % wl.tables[0].N
        idx.copy_(dev(ids))
        graph.replay()
        keep, wl.indices = wl.indices, ids
        assert_close(out.cpu().numpy(), oracle.forward_workload(wl), "out")
        counts = emb.grouping_counts()
        for t in range(2):
            lo, hi = wl.offsets[t * 128], wl.offsets[(t + 1) * 128]
            assert counts[t, 2] == len(np.unique(ids[lo:hi]))
        wl.indices = keep
    assert_close(emb.forward(dev(wl.indices), off, 128).cpu().numpy(), ref, "out")


def test_calls_go_to_the_current_stream(binding):  # noqa: F811
    import torch
    side = torch.cuda.Stream()
    for stream in (torch.cuda.default_stream(), side, torch.cuda.ExternalStream(side.cuda_stream)):
        with torch.cuda.stream(stream):
            assert binding._stream_ptr() == binding._stream_ptr(stream) == stream.cuda_stream


@pytest.mark.parametrize("big", [0, 2])
def test_cores_of_more_than_2_to_the_32_floats(binding, big):  # noqa: F811
    # first and last core of (2^25 + 64) slices of 128 floats, 17 GB; digits whose slices lie 2^32 floats apart
    n, r, most = [3, 2, 3], (1, 32, 8, 1) if big == 0 else (1, 8, 32, 1), (1 << 25) + 64
    n[big] = most
    used = [0, 5, 63, (1 << 25) - 1, 1 << 25, (1 << 25) + 5, most - 1]
    g = torch.Generator(device="cuda")
    g.manual_seed(big)
    cores = [torch.zeros((r[k], n[k], 4, r[k + 1]), device="cuda") for k in range(3)]
    for k in range(3):
        for i in used if k == big else range(n[k]):
            cores[k][:, i] = torch.randn((r[k], 4, r[k + 1]), generator=g, device="cuda")
    B = 70
    digits = [[used[b % len(used)] if k == big else (b + k) % n[k] for k in range(3)] for b in range(B)]
    ids = torch.tensor([(i * n[1] + j) * n[2] + m for i, j, m in digits], device="cuda")
    emb = binding.TTEmbeddingBag([int(np.prod(n, dtype=np.int64))], [n], [(4, 4, 4)], [r], B, B)
    emb.set_cores([cores])
    count, out = launches(binding, emb, ids, torch.arange(B + 1, device="cuda"), B)
    assert count == 1 and emb.status() == 0
    ref = torch.stack([torch.einsum("pa,aqb,bs->pqs", cores[0][0, i].double(), cores[1][:, j].double(), cores[2][:, m, :, 0].double()).reshape(-1)
                       for i, j, m in digits])
    assert_close(out.cpu().numpy(), ref.cpu().numpy(), "out")


R8, ANY = ((2, 4, 4), (1, 8, 8, 1)), ((3, 3, 5), (1, 6, 4, 1))


@pytest.mark.parametrize("shape,T,rows,B,lens,direct", [
    (R8, 8, 3000, 400, (1, 100), False), (R8, 8, 3_000_000, 400, (1, 100), True), (R8, 16, 3000, 4096, (1, 3), False), (R8, 4, 3000, 16_384, 1, False),
    (R8, 4, 3000, 4096, 1, True), (R8, 4, 60_000, 16_384, 1, True), (ANY, 1, 60_000, 20_000, (0, 5), True)])
def test_few_rows_are_shared(binding, shape, T, rows, B, lens, direct):  # noqa: F811
    n = (round(rows ** (1 / 3)) + 1,) * 3
    spec = TableSpec(N=rows, n=n, d=shape[0], r=shape[1], alpha=0.8, core_dist="normal", core_scale=0.4)
    wl = workloads.custom([spec] * T, B, lens, seed=T)
    emb = binding.from_workload(wl)
    count, out = launches(binding, emb, dev(wl.indices), dev(wl.offsets), B)
    assert (count == 1) == direct and emb.status() == 0
    assert_close(out.cpu().numpy(), oracle.forward_workload(wl, memo=True), "out")


def test_current_stream_without_the_raw_handle(binding, monkeypatch):  # noqa: F811
    # a torch that no longer has the call behind the shorter way
    side = torch.cuda.Stream()
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    for stream in (torch.cuda.default_stream(), side):
        with torch.cuda.stream(stream):
            assert binding._stream_ptr() == stream.cuda_stream


def test_stage_times(binding):  # noqa: F811
    # every stage of a forward has a time, as on the grouped path
    wl = build((4, 4, 4), (1, 8, 8, 1), 64, 2, 1, seed=13)
    times = []
    for backward in (False, True):
        emb = binding.from_workload(wl, enable_backward=backward)
        emb.enable_timing()
        emb.forward(dev(wl.indices), dev(wl.offsets), 64)
        times.append(emb.stage_ms())
        assert all(t >= 0 for t in times[-1].values())
    assert set(times[0]) == set(times[1]) >= {"grouping", "schedule", "contraction", "pooling", "k_sweep_fwd<2>"}
