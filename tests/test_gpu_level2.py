"""Level-2 products of four-core tables (P_2 = G_1[i_1] . G_2[i_2], stored for every level-2 node) at the ends of what a
table may be: first cores of 2^31 rows and more, few and many possible prefixes per present one.

Bar: max|err| <= 1e-5 * max|ref|, the bound of the other parity tests."""
import numpy as np
import pytest

from test_gpu_parity import TOL, binding  # noqa: F401  (binding: fixture)

pytestmark = pytest.mark.gpu


def rows_by_definition(cores, n, ids):
    """The rows of the ids in 64 bits, from device cores in slice-major layout [n][r_prev][d][r_next]."""
    digit, digits = ids, []
    for k in reversed(range(len(n))):
        digits.insert(0, digit % n[k])
        digit = digit // n[k]
    x = None
    for core, i in zip(cores, digits):
        s = core[i].double()
        x = s if x is None else (x.reshape(len(ids), -1, s.shape[1]) @ s.reshape(len(ids), s.shape[1], -1)).reshape(len(ids), 1, -1, s.shape[3])
    return x.reshape(len(ids), -1)


def handle(binding, n, d, r, lookups):  # noqa: F811
    import torch
    emb = binding.TTEmbeddingBag([int(np.prod(n))], [n], [d], [r], lookups, lookups, enable_backward=True)   # (grouped, however few lookups)
    shapes = [(r[k], n[k], d[k], r[k + 1]) for k in range(4)]
    g = torch.Generator(device="cuda").manual_seed(1)
    emb.set_cores([[torch.empty(s, device="cuda").normal_(generator=g) for s in shapes]])
    return emb, [c.view(n[k], r[k], d[k], r[k + 1]) for k, c in enumerate(emb.cores[0])]


def check(emb, cores, n, ids):
    import torch
    L = len(ids)
    out = emb.forward(ids, torch.arange(L + 1, device="cuda"), L)
    at_once = max(1, (1 << 26) // max(c[0].numel() for c in cores))   # half a gigabyte of slices in 64 bits
    want = torch.cat([rows_by_definition(cores, n, part) for part in ids.split(at_once)])
    err, scale = (out.double() - want).abs().max().item(), want.abs().max().item()
    assert err <= TOL * scale, (L, err, scale)
    assert emb.status() == 0


@pytest.mark.parametrize("n", [(33_554_432, 1, 2, 4), (34_000_000, 1, 2, 4)])   # 2^31 rows of 64, and some more
def test_first_core_of_2_to_the_31_rows(binding, n):  # noqa: F811
    import torch
    emb, cores = handle(binding, n, (64, 1, 1, 1), (1, 1, 1, 1, 1), 600_000)    # a first core of 8.6 GB
    for L in (500, 600_000):     # by node, by digit
        ids = torch.randint(0, int(np.prod(n)), (L,), device="cuda")
        ids[:2] = torch.tensor([0, int(np.prod(n)) - 1])
        check(emb, cores, n, ids)


# few and many lookups per possible prefix: by node (the last digits of every table) and by digit
@pytest.mark.parametrize("n,d,r", [
    ((1, 1, 3, 2), (1, 1, 1, 2), (1, 1, 1, 1, 1)),
    ((255, 3, 2, 2), (3, 2, 1, 2), (1, 5, 7, 3, 1)),          # odd rows and columns, just below, at and above one block
    ((256, 2, 2, 2), (2, 4, 4, 4), (1, 64, 64, 64, 1)),
    ((257, 1, 2, 2), (1, 3, 5, 2), (1, 33, 41, 3, 1)),        # two slices of columns, a second k pass of one
    ((3000, 1, 2, 2), (2, 2, 2, 2), (1, 4, 4, 4, 1)),         # several CTAs per second digit, several blocks
    ((2, 3000, 2, 2), (2, 2, 2, 2), (1, 4, 4, 4, 1)),
    ((40, 7, 2, 2), (128, 2, 1, 1), (1, 8, 16, 4, 1)),        # more than a tile of rows per prefix
    ((70, 5, 3, 2), (2, 8, 2, 1), (1, 128, 128, 6, 1)),
])
def test_rows(binding, n, d, r):  # noqa: F811
    import torch
    emb, cores = handle(binding, n, d, r, 50_000)
    for L in (1, 60, 50_000):
        check(emb, cores, n, torch.randint(0, int(np.prod(n)), (L,), device="cuda"))
    assert emb.check_guards() is None


def test_products_keep_32_bits(binding):  # noqa: F811
    # ranks of one and last cores of ones: a row is the product of two numbers, rounded once
    import torch
    n, d = (300, 7, 2, 2), (3, 5, 1, 1)
    emb, cores = handle(binding, n, d, (1, 1, 1, 1, 1), 8400)
    cores[2].fill_(1.0), cores[3].fill_(1.0)
    for L in (20, 8400):         # by node, by digit
        ids = torch.randperm(8400, device="cuda")[:L]
        out = emb.forward(ids, torch.arange(L + 1, device="cuda"), L)
        a, b = cores[0][ids // 28].reshape(L, 3, 1), cores[1][ids // 4 % 7].reshape(L, 1, 5)
        assert torch.equal(out, (a * b).reshape(L, 15)), L
