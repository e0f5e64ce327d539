"""BF16 and TF32 H_eff at links of at most 64 against the products in FP64 (numpy), and against the
general tensor-core kernel (tc_schedule 1): four and eight slices per unit, missing kinds, three-link
products, lists shorter and longer than one run per SM."""
import numpy as np
import pytest

from inputs import random_vector
from tests.gpu_util import dev, host, lib_and_ctx
from tests.test_gpu_dense import SLOTS, _abs, _apply, _problem

pytestmark = pytest.mark.gpu

CASES = [((16, 16, 16), (40, 30, 50), 0), ((16, 16, 16), (1, 0, 0), 1), ((32, 32, 32), (50, 45, 70), 12),
         ((48, 16, 64), (90, 0, 120), 3), ((64, 48, 32), (0, 60, 65), 0), ((64, 64, 64), (60, 61, 95), 24),
         ((16, 64, 48), (7, 3, 5), 9), ((64, 16, 16), (200, 3, 5), 0)]


@pytest.mark.parametrize("dtype,u", [(3, 2.0 ** -9), (2, 2.0 ** -10)])  # BF16; TF32, truncated between the stages
@pytest.mark.parametrize("shape,counts,nt", CASES)
def test_applications_within_rounding(shape, counts, nt, dtype, u):
    """At most six operand roundings per product (three-link ones: three operators, the input, two
    partial results; pair products four) and FP32 sums."""
    out = {}
    hint, pairs, triples = _problem(shape, counts, nt, sum(shape))
    n = 10 + sum(shape) + sum(counts[k] * (shape[p] + shape[q] + 2) for k, (p, q) in enumerate(SLOTS)) + \
        nt * (sum(shape) + 3)
    bound = (1 + u) ** 6 * (1 + n * 2.0 ** -24) - 1
    for schedule in (0, 1):
        attn, ctx = lib_and_ctx({"tc_schedule": schedule})
        keep = [[None if h is None else dev(h) for h in hint], {k: (dev(a), dev(b)) for k, (a, b) in pairs.items()},
                None if triples is None else tuple(dev(t) for t in triples)]
        H = attn.attn_heff_create(ctx, shape, *keep)
        for rep in (0, 1):
            x = random_vector(shape, 100 + rep)
            y = dev(np.full(shape, np.nan))
            attn.attn_heff_apply(H, dev(x), y, dtype)
            attn.attn_sync(ctx)
            ref = _apply(hint, pairs, triples, x)
            absref = _apply([_abs(h) for h in hint], {k: _abs(v) for k, v in pairs.items()}, _abs(triples), np.abs(x))
            assert np.all(np.abs(host(y) - ref) <= bound * absref), (schedule, rep)
        out[schedule] = host(y)
        attn.attn_heff_destroy(H)
        attn.attn_destroy(ctx)
    # the same roundings in both kernels: they differ by the order of FP32 sums
    assert np.linalg.norm(out[0] - out[1]) <= 1e-5 * np.linalg.norm(out[1])
