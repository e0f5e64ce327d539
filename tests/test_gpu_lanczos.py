"""Lanczos at vector lengths around the one-launch step: fewer entries than CTAs, lengths that
divide over nothing, the largest that fits the cluster and one beyond it. Start and operator are such
that the Krylov space is exhausted or converged within the depth, so the lowest pair is that of the
dense operator."""
import numpy as np
import pytest

from inputs import random_operators, random_vector
from tests.gpu_util import dev, host, lib_and_ctx

pytestmark = pytest.mark.gpu


def _heff(attn, ctx, shape, seed, bias):
    """Internal operators with one low direction each (a gap of `bias`) and weak pair products."""
    hint = [random_operators(1, m, seed, 10 + s)[0] * 0.3 for s, m in enumerate(shape)]
    low = [np.ones(m) / np.sqrt(m) for m in shape]
    for s in range(3):
        hint[s] -= bias * np.outer(low[s], low[s])
    pairs = {k: (0.2 * random_operators(3, shape[p], seed, 20 + k), random_operators(3, shape[q], seed, 30 + k))
             for k, (p, q) in enumerate(((0, 1), (0, 2), (1, 2)))}
    H = attn.attn_heff_create(ctx, shape, [dev(h) for h in hint], {k: (dev(a), dev(b)) for k, (a, b) in pairs.items()})
    start = np.einsum("a,b,c->abc", *low) + 0.02 * random_vector(shape, 7)
    return H, start


def _residual(attn, H, v, theta):
    y = attn.attn_heff_apply_host(H, v)
    return np.linalg.norm(y - theta * v)


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 2, 1), (2, 2, 4), (3, 5, 7), (17, 16, 15), (16, 16, 16), (20, 31, 33),
                                   (27, 28, 27), (28, 28, 28)])
@pytest.mark.parametrize("graph", [0, 1])
def test_lowest_pair(shape, graph):
    attn, ctx = lib_and_ctx({"lanczos_depth": 50 if np.prod(shape) < 6000 else 24, "use_graphs": graph,
                             "lanczos_tol": 1e-13 if graph == 0 else 0.0})
    H, start = _heff(attn, ctx, shape, int(sum(shape)), 6.0)
    for rep in range(2):
        t = dev(start)
        theta, iters = attn.attn_eigsolve(H, t)
        v = host(t)
        assert abs(np.linalg.norm(v) - 1.0) < 1e-13
        # the Ritz value is the Rayleigh quotient of the vector (FP64), and its residual small: a
        # gap of about 6 - 2 against a spread below 30 converges by a factor of at least 2 a step
        assert abs(float((v * attn.attn_heff_apply_host(H, v)).sum()) - theta) <= 1e-12 * abs(theta)
        assert _residual(attn, H, v, theta) <= 30.0 * 2.0 ** -min(20, int(np.prod(shape)) * 20)
    if np.prod(shape) <= 300:
        e = np.eye(int(np.prod(shape))).reshape(-1, *shape)
        dense = np.stack([attn.attn_heff_apply_host(H, b).ravel() for b in e])
        w, u = np.linalg.eigh(0.5 * (dense + dense.T))
        assert abs(theta - w[0]) <= 1e-12 * abs(w[0])
        if len(w) > 1:
            assert abs(abs(u[:, 0] @ v.ravel()) - 1.0) < 1e-10
    attn.attn_heff_destroy(H)
    attn.attn_destroy(ctx)
