"""Device memory of the dense pair operators, as a caller's allocator sees it."""
import contextlib

import numpy as np
import pytest

from inputs import random_operators, random_vector
from tests.gpu_util import dev, host, lib_and_ctx

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _allocator(alloc):
    import torch
    from paper_2507_21236_gb300 import attn

    attn.attn_set_allocator(alloc, lambda p, n, device: torch.cuda.caching_allocator_delete(p))
    try:
        yield
    finally:
        attn.attn_set_allocator(None, None)


def _pair01(shape, R, seed):
    return {0: tuple(dev(random_operators(R, shape[s], seed, 20 + s, symmetric=False)) for s in (0, 1))}


def test_split_operators_are_made_within_a_gigabyte():
    """A second link without factors of two: M (12769 x 12769, 1.3 GB) is made in parts of whole
    slices tiles, which begin and end inside a value of the first link, and only its slices (2 GB)
    are a block above 1 GiB. Applications before and after agree within the split path's 1e-12."""
    import torch

    sizes = []

    def alloc(n, device):
        sizes.append(n)
        return torch.cuda.caching_allocator_alloc(n, device)

    shape, R = (113, 113, 16), 160
    with _allocator(alloc):
        attn, ctx = lib_and_ctx({"f64_split": 1})
        hint = [dev(random_operators(1, shape[s], 4, 10 + s)[0]) for s in range(3)]
        H = attn.attn_heff_create(ctx, shape, hint, _pair01(shape, R, 4))
        x = dev(random_vector(shape, 1))
        out = []
        for _ in range(4):
            y = dev(np.full(shape, np.nan))
            attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
            attn.attn_sync(ctx)
            out.append(host(y))
        attn.attn_heff_destroy(H)
        attn.attn_destroy(ctx)
    assert not np.array_equal(out[3], out[0])  # the sums were made
    assert np.abs(out[3] - out[0]).max() <= 1e-12 * np.abs(out[0]).max()
    big = [n for n in sizes if n > 1 << 30]
    assert len(big) == 1 and big[0] > 12 * 12769 ** 2, big


@pytest.mark.parametrize("split", [0, 1])
def test_refused_memory_is_asked_for_ever_more_rarely(split):
    """An allocator that refuses the operators' memory for 40 applications: the first attempts follow
    one another, later ones wait for 1, 2, 4 .. applications, and every application goes product by
    product to the same bits. Once memory is there an application within the longest wait takes the sums."""
    import torch

    shape, R, limit = ((64, 64, 64), 60, 1 << 29) if split else ((32, 32, 32), 40, 20000000)
    refuse, attempts = [True], []

    def alloc(n, device):
        if refuse[0] and n >= limit:
            attempts.append(n)
            return 0
        return torch.cuda.caching_allocator_alloc(n, device)

    with _allocator(alloc):
        attn, ctx = lib_and_ctx({"f64_split": split})
        pairs = {k: tuple(dev(random_operators(R, shape[s], 5, 20 + 2 * k + i, symmetric=False))
                          for i, s in enumerate(slots)) for k, slots in enumerate(((0, 1), (0, 2), (1, 2)))}
        H = attn.attn_heff_create(ctx, shape, (None, None, None), pairs)
        x = dev(random_vector(shape, 1))
        y = dev(np.empty(shape))
        attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
        first = host(y)
        for _ in range(39):
            attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
        assert np.array_equal(host(y), first)
        assert 4 <= len(attempts) <= 10
        refuse[0] = False
        for _ in range(65):
            attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
        assert not np.array_equal(host(y), first)
        assert np.abs(host(y) - first).max() <= 1e-12 * np.abs(first).max()
        attn.attn_heff_destroy(H)
        attn.attn_destroy(ctx)
