"""Performance cases of the TT embedding bag: calls that programs which use it make, over the shapes they make them with.

A case is one handle (`TTEmbeddingBag`: tables, dim factors, ranks, batch, bag lengths) and one direction:

* ``forward``    one pooled look-up, as in inference;
* ``gradients``  forward, then the gradients of all cores (`backward`), as a replica that reduces gradients before updating;
* ``step``       forward, then backward and SGD update in one call (`backward_sgd`), the single-GPU training step.

Row ids follow a bounded power law; popular ids are the small ones (``identity``) or spread over the table (``scattered``,
as after hashing).  Tables have log-uniform row counts.  `grad_out` is that of a loss averaged over the batch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_03459_b200.binding import TTEmbeddingBag

LR = 0.05

_BASE = {
    "tables": 8, "rows_lo": 10_000, "rows_hi": 40_000_000, "dims": "4x4x4", "ranks": "16", "batch": 4096,
    "bag_lo": 1, "bag_hi": 100, "bags_per_table": False, "alpha_lo": 0.8, "alpha_hi": 1.2, "mapping": "identity",
    "ids": "int64", "pool": "sum", "mode": "forward", "core_std": 0.05, "shapes": 3,
}


def _case(name=None, **fields):
    c = dict(_BASE)
    c.update(fields)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one table, 1024 single look-ups; launches and latency are all there is
        _case("one-table-1024", tables=1, rows_lo=1_000_000, rows_hi=1_000_000, dims="4x4x4", ranks="8", batch=1024, bag_hi=1,
              alpha_lo=1.05, alpha_hi=1.05),
        # an online inference request over eight tables of production size, 32-bit ids, hashed rows
        _case("request-8-tables", tables=8, ranks="16", batch=96, bag_hi=20, ids="int32", mapping="scattered"),
        # batch inference on one wide table (D = 128), fixed bags of twenty
        _case("wide-table", tables=1, rows_lo=10_000_000, rows_hi=10_000_000, dims="4x8x4", ranks="32", batch=32768, bag_lo=20,
              bag_hi=20, alpha_lo=1.1, alpha_hi=1.1),
        # four cores with rank 64, deep shared prefixes: inference
        _case("four-cores", tables=1, rows_lo=16_777_216, rows_hi=16_777_216, dims="2x4x4x4", ranks="64", batch=65536, bag_lo=8,
              bag_hi=8, alpha_lo=1.2, alpha_hi=1.2, core_std=0.02),
        # the same table in training
        _case("four-cores-training", tables=1, rows_lo=16_777_216, rows_hi=16_777_216, dims="2x4x4x4", ranks="64", batch=8192,
              bag_lo=8, bag_hi=8, alpha_lo=1.2, alpha_hi=1.2, core_std=0.02, mode="gradients"),
        # recommender inference at full batch: sixty tables of ranks 16 and 32
        _case("sixty-tables", tables=60, ranks="16|32", batch=32768),
        # the training step on those tables
        _case("sixty-tables-step", tables=60, ranks="16|32", batch=32768, mode="step"),
        # hundreds of tables, most with short bags, D = 32: the training step
        _case("many-tables-step", tables=240, dims="2x4x4", ranks="32", batch=32768, bag_hi=64, bags_per_table=True, mode="step",
              shapes=6),
        # an ordinary data-parallel replica's share: eight tables, batch 4096, gradients for the all-reduce
        _case("replica-gradients", tables=8, ranks="16", batch=4096, mode="gradients"),
        # factors of no round size (D = 45, ranks 6 and 4), odd batch
        _case("odd-factors", tables=4, dims="3x3x5", ranks="6,4", batch=5003, mode="gradients"),
        # narrow rows, per-lookup weights, 32-bit ids, odd batch: training
        _case("weighted-narrow", tables=8, dims="2x2x4", ranks="16", batch=10007, ids="int32", pool="weighted", mode="gradients"),
        # mean pooling over short bags, some of them empty, hashed rows: training
        _case("mean-short-bags", tables=4, dims="2x4x4", ranks="8", batch=65536, bag_lo=0, bag_hi=4, pool="mean",
              mapping="scattered", mode="gradients"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    dims, ranks = rng.choice([
        ("4x4x4", "8"), ("4x4x4", "16"), ("4x4x4", "32"), ("4x4x4", "16|32"), ("2x4x4", "8"), ("2x4x4", "16"), ("2x4x4", "32"),
        ("2x2x4", "8"), ("2x2x4", "16"), ("2x2x4", "32"), ("4x8x4", "32"), ("2x4x4x4", "64"), ("3x3x5", "6,4"), ("8x8", "24")])
    c = _case(dims=dims, ranks=ranks, mode=rng.choice(["forward", "gradients", "step"]), shapes=rng.randrange(1, 1000),
              mapping=rng.choice(["identity", "identity", "scattered"]), ids=rng.choice(["int64", "int64", "int32"]),
              pool=rng.choice(["sum", "sum", "sum", "mean", "weighted"]), batch=log_int(64, 65536))
    odd = dims in ("3x3x5", "8x8")          # cores of such tables are returned one by one
    c["tables"] = log_int(1, 6) if odd else log_int(1, 64)
    c["bag_lo"], c["bag_hi"] = rng.choice([(1, 1), (1, 100), (1, 20), (0, 5), (8, 8)])
    if dims == "2x4x4x4":
        c["core_std"] = 0.02
        c["tables"] = min(c["tables"], 4)
        c["batch"] = min(c["batch"], 8192) if c["mode"] != "forward" else c["batch"]
    if dims == "8x8":
        c["rows_hi"] = 4_000_000
    mean_bag = 0.5 * (c["bag_lo"] + c["bag_hi"])
    most = 4_000_000 if odd or dims == "2x4x4x4" else 24_000_000   # lookups: below the largest listed case's work
    c["batch"] = max(1, min(c["batch"], int(most / (c["tables"] * mean_bag))))
    return c


# ------------------------------------------------------------------------------------------------ tables of a case
def _tables(case):
    """Row counts, row factors, dim factors, ranks and power-law exponents of the case's tables."""
    rng = np.random.default_rng(case["shapes"])
    dims = tuple(int(x) for x in case["dims"].split("x"))
    K = len(dims)
    found = []
    for _ in range(case["tables"]):
        N = int(round(10.0 ** rng.uniform(math.log10(case["rows_lo"]), math.log10(case["rows_hi"]))))
        n = max(1, int(round(N ** (1.0 / K))))
        while n ** K < N:
            n += 1
        while n > 1 and (n - 1) ** K >= N:
            n -= 1
        factors = (-(-N // n ** (K - 1)),) + (n,) * (K - 1)
        if "|" in case["ranks"]:
            inner = tuple(int(rng.choice([int(x) for x in case["ranks"].split("|")])) for _ in range(K - 1))
        elif "," in case["ranks"]:
            inner = tuple(int(x) for x in case["ranks"].split(","))
        else:
            inner = (int(case["ranks"]),) * (K - 1)
        alpha = float(rng.uniform(case["alpha_lo"], case["alpha_hi"]))
        longest = int(round(case["bag_hi"] ** rng.uniform())) if case["bags_per_table"] else case["bag_hi"]
        found.append({"N": N, "n": factors, "d": dims, "r": (1,) + inner + (1,), "alpha": alpha, "longest": longest})
    return found


def _core_shapes(t):
    return [(t["r"][k], t["n"][k], t["d"][k], t["r"][k + 1]) for k in range(len(t["n"]))]


def _spread(N):
    """Multiplier that spreads popularity ranks over the row ids (coprime to N)."""
    a = max(2, 2654435761 % N)
    while math.gcd(a, N) != 1:
        a += 1
    return a


def _inputs(case, seed):
    """Cores (index order [r_prev, n, d, r_next]), ids, offsets, weights and grad_out on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    tables, B = _tables(case), case["batch"]
    cores = [[torch.randn(s, generator=g, device="cuda") * case["core_std"] for s in _core_shapes(t)] for t in tables]
    lens = torch.cat([torch.randint(case["bag_lo"], t["longest"] + 1, (B,), generator=g, device="cuda") for t in tables])
    offsets = torch.zeros(len(tables) * B + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offsets[1:])
    counts = lens.view(len(tables), B).sum(1).tolist()
    L = sum(counts)
    ids = torch.empty(L, dtype=torch.int64 if case["ids"] == "int64" else torch.int32, device="cuda")
    at = 0
    for t, n in zip(tables, counts):
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        e = 1.0 - t["alpha"]
        lo, hi = 0.5 ** e, (t["N"] + 0.5) ** e
        rank = (u.mul_(hi - lo).add_(lo)).pow_(1.0 / e).add_(0.5).floor_().to(torch.int64).clamp_(1, t["N"]).sub_(1)
        if case["mapping"] == "scattered":
            rank.mul_(_spread(t["N"])).remainder_(t["N"])
        ids[at:at + n] = rank
        at += n
    weights = grad = None
    if case["pool"] == "weighted":
        weights = torch.rand(L, generator=g, device="cuda") + 0.5
    if case["mode"] != "forward":
        D = math.prod(tables[0]["d"])
        grad = torch.randn((B, len(tables) * D), generator=g, device="cuda") / B
    return tables, cores, ids, offsets, weights, grad


# ------------------------------------------------------------------------------------------------ one pass
def prepare(case, seed):
    tables, cores, ids, offsets, weights, grad = _inputs(case, seed)
    emb = TTEmbeddingBag([t["N"] for t in tables], [t["n"] for t in tables], [t["d"] for t in tables], [t["r"] for t in tables],
                         case["batch"], max(ids.numel(), 1), enable_backward=case["mode"] != "forward",
                         enable_weighted=case["pool"] != "sum")
    emb.set_cores(cores)
    emb.set_pooling("mean" if case["pool"] == "mean" else "sum", weights)
    out = torch.empty((case["batch"], emb.T * emb.D), dtype=torch.float32, device="cuda")
    return {"emb": emb, "ids": ids, "offsets": offsets, "batch": case["batch"], "grad": grad, "mode": case["mode"], "out": out,
            "flat": _flat(tables)}


def _flat(tables):
    """Whether the cores fill one flat buffer without gaps (each is a multiple of four floats)."""
    return all(math.prod(s) % 4 == 0 for t in tables for s in _core_shapes(t))


def run(state):
    emb = state["emb"]
    out = {"out": emb.forward(state["ids"], state["offsets"], state["batch"], out=state["out"])}
    if state["mode"] == "gradients":
        grads = emb.backward(state["grad"])
        out["grads"] = emb.flat_grads if state["flat"] else grads
    elif state["mode"] == "step":
        grads = emb.backward_sgd(state["grad"], LR)
        out["grads"] = emb.flat_grads if state["flat"] else grads
        out["cores"] = emb.flat_cores if state["flat"] else emb.cores
    return out


# ------------------------------------------------------------------------------------------------ work and tolerance
def _mass(t, k):
    """Probability that a look-up's popularity rank is at most k."""
    e = 1.0 - t["alpha"]
    return ((k + 0.5) ** e - 0.5 ** e) / ((t["N"] + 0.5) ** e - 0.5 ** e)


def _distinct(t, L, mapping):
    """Expected number of distinct length-k prefixes (k = 1..K) among L look-ups of the table."""
    K, N = len(t["n"]), t["N"]
    edges = np.unique(np.concatenate([np.arange(0, min(N, 2000)), np.geomspace(max(1, min(N, 2000)), N, 4000).astype(np.int64), [N]])).astype(np.float64)
    size, mass = np.diff(edges), np.diff(_mass(t, edges))
    rows = float(np.sum(size * -np.expm1(-L * mass / size)))
    found = []
    for k in range(1, K):
        below = math.prod(t["n"][k:])
        count = -(-N // below)
        if mapping == "identity":
            cuts = np.minimum(np.arange(count + 1, dtype=np.float64) * below, N)
            found.append(float(np.sum(-np.expm1(-L * np.diff(_mass(t, cuts))))))
        else:
            found.append(count * -math.expm1(-rows / count))
    return found + [rows]


def work(case):
    tables, B, T = _tables(case), case["batch"], case["tables"]
    D = math.prod(tables[0]["d"])
    train = case["mode"] != "forward"
    lookups = flops = floats = 0.0
    for t in tables:
        L = B * 0.5 * (case["bag_lo"] + t["longest"])
        lookups += L
        floats += sum(math.prod(s) for s in _core_shapes(t))
        found, width = _distinct(t, L, case["mapping"]), t["d"][0]
        flops += (L * D + (L * D if train else 0)) * (2 if case["pool"] == "weighted" else 1)
        for k in range(1, len(t["n"])):
            products = 2.0 * found[k] * width * t["r"][k] * t["d"][k] * t["r"][k + 1]   # one product per distinct prefix
            flops += products * (3 if train else 1)                                     # and two for its gradients
            width *= t["d"][k]
    bytes_ = lookups * (8 if case["ids"] == "int64" else 4) + 8 * (T * B + 1) + 4 * floats + 4 * B * T * D
    if case["pool"] == "weighted":
        bytes_ += 4 * lookups
    if train:
        bytes_ += 4 * B * T * D + 4 * floats + (4 * floats if case["mode"] == "step" else 0)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # fp32 sums and products split into three tensor-core terms; against 64 bits at most 5.3e-7 (out) and 2.2e-6 (gradients),
    # the same inputs twice 1.3e-6 and single values 5.9e-5
    return {"rel": 1e-5, "max": 4e-4}


# ------------------------------------------------------------------------------------------------ 64-bit results
def exact(case, seed):
    tables, cores, ids, offsets, weights, grad = _inputs(case, seed)
    B, D = case["batch"], math.prod(tables[0]["d"])
    out = torch.zeros((B, len(tables) * D), dtype=torch.float64, device="cuda")
    all_grads, all_cores = [], []
    ends = offsets[::B].tolist()
    for t, table in enumerate(tables):
        G = [c.double().movedim(1, 0).contiguous() for c in cores[t]]                 # [n, r_prev, d, r_next]
        off = offsets[t * B:(t + 1) * B + 1] - ends[t]
        lens = off[1:] - off[:-1]
        bag = torch.repeat_interleave(torch.arange(B, device="cuda"), lens)
        rows, slot = torch.unique(ids[ends[t]:ends[t + 1]].long(), return_inverse=True)
        factor = None
        if weights is not None:
            factor = weights[ends[t]:ends[t + 1]].double()
        elif case["pool"] == "mean":
            factor = 1.0 / lens[bag].double()
        # distinct prefixes, shortest first; up[k]: the parent of each node of level k
        vals, up = [rows], []
        for n in reversed(table["n"][1:]):
            prefix, parent = torch.unique(vals[0] // n, return_inverse=True)
            vals.insert(0, prefix)
            up.insert(0, parent)
        digit = [vals[0]] + [v % n for v, n in zip(vals[1:], table["n"][1:])]
        P = [G[0][digit[0]].reshape(vals[0].numel(), table["d"][0], table["r"][1])]
        for k in range(1, len(G)):
            P.append(torch.cat([(P[k - 1][p] @ G[k][i].flatten(2)).reshape(i.numel(), -1, table["r"][k + 1])
                                for i, p in zip(digit[k].split(8192), up[k - 1].split(8192))]))
        E = P[-1].reshape(rows.numel(), D)
        block = out[:, t * D:(t + 1) * D]
        for i in range(0, slot.numel(), 1 << 20):
            x = E[slot[i:i + (1 << 20)]]
            block.index_add_(0, bag[i:i + (1 << 20)], x if factor is None else x * factor[i:i + (1 << 20), None])
        if grad is None:
            continue
        dE = torch.zeros_like(E)
        g = grad[:, t * D:(t + 1) * D].double()
        for i in range(0, slot.numel(), 1 << 20):
            x = g[bag[i:i + (1 << 20)]]
            dE.index_add_(0, slot[i:i + (1 << 20)], x if factor is None else x * factor[i:i + (1 << 20), None])
        dG, d = [torch.zeros_like(x) for x in G], dE
        for k in range(len(G) - 1, 0, -1):
            below = torch.zeros_like(P[k - 1])
            d = d.reshape(vals[k].numel(), P[k - 1].shape[1], -1)
            for i, p, x in zip(digit[k].split(8192), up[k - 1].split(8192), d.split(8192)):
                dG[k].flatten(2).index_add_(0, i, P[k - 1][p].mT @ x)
                below.index_add_(0, p, x @ G[k][i].flatten(2).mT)
            d = below
        dG[0].index_add_(0, digit[0], d.reshape(vals[0].numel(), 1, table["d"][0], table["r"][1]))
        all_grads.append([x.flatten() for x in dG])
        all_cores.append([(x - LR * y).flatten() for x, y in zip(G, dG)])
    result = {"out": out}
    if grad is not None:
        flat = _flat(tables)
        result["grads"] = torch.cat([x for t in all_grads for x in t]) if flat else all_grads
        if case["mode"] == "step":
            result["cores"] = torch.cat([x for t in all_cores for x in t]) if flat else all_cores
    return result
