"""attn_profile_read counts 2 m_l V FLOPs per operator applied, whatever way an FP64 application goes:
product by product at first, through the sums of the pairs' products later, and in the application
that makes the sums."""
import numpy as np
import pytest

from inputs import random_operators, random_vector
from tests.gpu_util import dev, lib_and_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,counts,nt,split", [((16, 24, 20), (12, 0, 14), 0, 0), ((32, 32, 32), (40, 45, 50), 2, 0),
                                                   ((64, 64, 64), (60, 2, 55), 0, 1), ((64, 64, 64), (140, 130, 150), 0, 1)])
def test_fp64_application_counts_its_products(shape, counts, nt, split):
    attn, ctx = lib_and_ctx({"f64_split": split})
    hint = [None, dev(random_operators(1, shape[1], 3, 11)[0]), dev(random_operators(1, shape[2], 3, 12)[0])]
    pairs = {k: tuple(dev(random_operators(counts[k], shape[s], 3, 20 + 2 * k + i, symmetric=False))
                      for i, s in enumerate(slots)) for k, slots in enumerate(((0, 1), (0, 2), (1, 2))) if counts[k]}
    triples = tuple(dev(random_operators(nt, shape[s], 3, 30 + s, symmetric=False)) for s in range(3)) if nt else None
    H = attn.attn_heff_create(ctx, shape, hint, pairs, triples)
    flops = attn.attn_heff_info(H)[2]
    x, y = dev(random_vector(shape, 1)), dev(np.empty(shape))
    records = set()
    for rep in range(4):
        attn.attn_profile_enable(ctx)
        attn.attn_heff_apply(H, x, y, attn.ATTN_F64)
        rec = [attn.attn_profile_read(ctx, kid) for kid in (1, 3)]
        records.add(sum(r[1] for r in rec))
        assert abs(sum(r[2] for r in rec) / flops - 1.0) <= 1e-12, rep
    assert len(records) > 1  # more than one way was taken
    attn.attn_profile_enable(ctx, False)
    attn.attn_heff_destroy(H)
    attn.attn_destroy(ctx)
