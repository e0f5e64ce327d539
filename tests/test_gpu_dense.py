"""H_eff through one dense operator per link pair against the products applied one by one in
FP64 (numpy), for every application of a handle: the first ones go product by product, later
ones through the sums."""
import numpy as np
import pytest

from inputs import random_operators, random_vector
from tests.gpu_util import dev, host, lib_and_ctx

pytestmark = pytest.mark.gpu

SUB = ("ia,jb,abc->ijc", "ia,jc,abc->ibj", "ib,jc,abc->aij")
SLOTS = ((0, 1), (0, 2), (1, 2))
MODE = ("ia,abc->ibc", "ib,abc->aic", "ic,abc->abi")


def _problem(shape, counts, nt, seed):
    hint = [random_operators(1, shape[s], seed, 10 + s)[0] if (seed + s) % 4 else None for s in range(3)]
    pairs = {k: tuple(random_operators(counts[k], shape[s], seed, 20 + 2 * k + i, symmetric=False)
                      for i, s in enumerate(SLOTS[k])) for k in range(3) if counts[k]}
    triples = tuple(random_operators(nt, shape[s], seed, 30 + s, symmetric=False) for s in range(3)) if nt else None
    return hint, pairs, triples


def _apply(hint, pairs, triples, x):
    y = np.zeros_like(x)
    for s in range(3):
        if hint[s] is not None:
            y += np.einsum(MODE[s], hint[s], x)
    for k, (a, b) in pairs.items():
        for r in range(len(a)):
            y += np.einsum(SUB[k], a[r], b[r], x, optimize=True)
    if triples is not None:
        for r in range(len(triples[0])):
            y += np.einsum("ia,jb,kc,abc->ijk", triples[0][r], triples[1][r], triples[2][r], x, optimize=True)
    return y


def _abs(t):
    if t is None:
        return None
    return np.abs(t) if isinstance(t, np.ndarray) else tuple(np.abs(v) for v in t)


# block edges (4 and 8 wide), K steps of 64 and 128, single rows, missing kinds, triples, every block size
CASES = [((2, 2, 4), (3, 2, 5), 0), ((4, 4, 16), (9, 0, 7), 2), ((16, 16, 16), (12, 12, 14), 0),
         ((5, 7, 9), (11, 30, 8), 3), ((1, 33, 17), (20, 0, 40), 0), ((32, 31, 33), (40, 45, 50), 1),
         ((24, 48, 40), (70, 1, 65), 0), ((64, 72, 80), (90, 100, 80), 0)]


@pytest.mark.parametrize("shape,counts,nt", CASES)
def test_repeated_fp64_applications_match_products(shape, counts, nt):
    attn, ctx = lib_and_ctx()
    seed = sum(shape)
    hint, pairs, triples = _problem(shape, counts, nt, seed)
    keep = [[None if h is None else dev(h) for h in hint], {k: (dev(a), dev(b)) for k, (a, b) in pairs.items()},
            None if triples is None else tuple(dev(t) for t in triples)]
    H = attn.attn_heff_create(ctx, shape, *keep)
    # every path sums at most this many products per output, each with rounded factors
    n = 3 + sum(shape) + sum(counts[k] * (shape[p] + shape[q] + 2) + shape[p] * shape[q]
                             for k, (p, q) in enumerate(SLOTS)) + nt * (sum(shape) + 3)
    for rep in range(4):
        x = random_vector(shape, 100 + rep)
        y = dev(np.full(shape, np.nan))
        attn.attn_heff_apply(H, dev(x), y, attn.ATTN_F64)
        ref = _apply(hint, pairs, triples, x)
        absref = _apply([_abs(h) for h in hint], {k: _abs(v) for k, v in pairs.items()}, _abs(triples), np.abs(x))
        assert np.all(np.abs(host(y) - ref) <= 2 * n * 2.0 ** -53 * absref), rep
    attn.attn_heff_destroy(H)
    attn.attn_destroy(ctx)


@pytest.mark.parametrize("shape,counts", [((64, 64, 64), (140, 130, 150)), ((48, 56, 72), (120, 0, 110)),
                                          ((33, 40, 130), (60, 300, 90)), ((16, 24, 20), (12, 12, 14))])
def test_repeated_split_applications_match_products(shape, counts):
    """f64_split: every application within the split path's tolerance (1e-12 of the largest
    entry); zero rows of operators and of x stay exact zeros."""
    attn, ctx = lib_and_ctx({"f64_split": 1})
    _, pairs, _ = _problem(shape, counts, 0, sum(shape))
    hint = [None, random_operators(1, shape[1], 3, 11)[0], None]
    for k, (p, q) in enumerate(SLOTS):
        if k in pairs:
            for t, s in zip(pairs[k], (p, q)):
                if s == 0:
                    t[:, 5, :] = 0.0
    keep = [[None if h is None else dev(h) for h in hint], {k: (dev(a), dev(b)) for k, (a, b) in pairs.items()}]
    H = attn.attn_heff_create(ctx, shape, *keep)
    for rep in range(3):
        x = random_vector(shape, 100 + rep)
        x[5] = 0.0
        y = dev(np.full(shape, np.nan))
        attn.attn_heff_apply(H, dev(x), y, attn.ATTN_F64)
        attn.attn_sync(ctx)
        ref = _apply(hint, pairs, None, x)
        got = host(y)
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), rep
        if counts[2] == 0:
            assert np.all(got[5] == 0.0)
    attn.attn_heff_destroy(H)
    attn.attn_destroy(ctx)


def test_split_application_without_memory_for_the_sums():
    """A device allocator that refuses the slices (604 MB), their exponents (under 1 MB) or the
    stage they are made in (134 MB): the application goes product by product as the first one did, bit
    for bit, and takes the sums once memory is there."""
    import torch
    from paper_2507_21236_gb300 import attn as A_

    refuse, refused = [0, 0], []

    def alloc(n, device):
        if refuse[0] <= n < refuse[1]:
            refused.append(n)
            return 0
        return torch.cuda.caching_allocator_alloc(n, device)

    shape, counts = (64, 64, 64), (60, 50, 55)
    hint, pairs, _ = _problem(shape, counts, 0, 7)
    x = dev(random_vector(shape, 100))
    A_.attn_set_allocator(alloc, lambda p, n, device: torch.cuda.caching_allocator_delete(p))
    try:
        attn, ctx = lib_and_ctx({"f64_split": 1})
        keep = [[None if h is None else dev(h) for h in hint], {k: (dev(a), dev(b)) for k, (a, b) in pairs.items()}]
        H = attn.attn_heff_create(ctx, shape, *keep)
        out = []
        for sizes in ((0, 0), (1 << 29, 1 << 40), (0, 1 << 20), (130000000, 1 << 29), (0, 0)):
            refuse[:] = sizes
            refused.clear()
            y = dev(np.full(shape, np.nan))
            attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
            attn.attn_sync(ctx)
            out.append(host(y))
            assert bool(refused) == bool(refuse[1])
        attn.attn_heff_destroy(H)
        attn.attn_destroy(ctx)
    finally:
        A_.attn_set_allocator(None, None)
    for y in out[1:4]:
        assert np.array_equal(y, out[0])
    assert np.abs(out[4] - out[0]).max() <= 1e-12 * np.abs(out[0]).max()
    assert not np.array_equal(out[4], out[0])
