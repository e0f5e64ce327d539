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


def _bound(V, depth, theta):
    """Residual after `depth` steps: of the start's part outside the lowest state (0.02 sqrt(V)) each step
    keeps exp(-2 asinh sqrt(gap / spread)), gap above 4 (6 less what the weak operators shift it by) of a
    spectrum below 20 wide; and the rounding of the recurrence."""
    rate = np.exp(-2.0 * np.arcsinh(np.sqrt(4.0 / 20.0)))
    return 2.0 * 24.0 * 0.02 * np.sqrt(V) * rate ** (depth - 1) + 1e-12 * abs(theta)


# 16 CTAs with ceil(V / 16) entries of depth + 1 vectors in 200 KB each: V = 16384 at depth 24 and 19500
# at depth 20 are the largest that fit, 16275 leaves the last CTA short, the others are beyond it
@pytest.mark.parametrize("shape,depth", [((16, 32, 32), 24), ((16, 32, 33), 24), ((15, 31, 35), 24), ((25, 26, 30), 20),
                                         ((25, 26, 31), 20)])
@pytest.mark.parametrize("graph", [0, 1])
def test_lowest_pair_at_the_limit_of_the_cluster(shape, depth, graph):
    attn, ctx = lib_and_ctx({"lanczos_depth": depth, "use_graphs": graph, "lanczos_tol": 0.0})
    H, start = _heff(attn, ctx, shape, int(sum(shape)), 6.0)
    for rep in range(2):
        t = dev(start)
        theta, iters = attn.attn_eigsolve(H, t)
        assert iters == depth
        v = host(t)
        assert abs(np.linalg.norm(v) - 1.0) < 1e-13
        assert abs(float((v * attn.attn_heff_apply_host(H, v)).sum()) - theta) <= 1e-12 * abs(theta)
        assert _residual(attn, H, v, theta) <= _bound(np.prod(shape), depth, theta)
    attn.attn_heff_destroy(H)
    attn.attn_destroy(ctx)


@pytest.mark.parametrize("shape,depth", [((16, 16, 16), 24), ((32, 32, 32), 24), ((32, 32, 48), 24), ((32, 32, 32), 20)])
def test_fp32_basis_at_the_limit_of_the_cluster(shape, depth):
    """TF32 matvecs: 32768 entries are the largest whose FP32 basis fits at depth 24. The Ritz value agrees
    with the FP64 basis's to the FP32 rounding of each of the basis vectors. (No residual: the operator
    rounds its input to TF32, so on the Ritz vector it is not the sum of what it gave on the basis.)"""
    out = {}
    for basis in (0, 1):
        attn, ctx = lib_and_ctx({"lanczos_depth": depth, "lanczos_tol": 0.0, "matvec_dtype": 2, "refine_steps": 0,
                                 "lanczos_basis": basis})
        H, start = _heff(attn, ctx, shape, int(sum(shape)), 6.0)
        t = dev(start)
        theta, _ = attn.attn_eigsolve(H, t)
        v = host(t)
        assert abs(np.linalg.norm(v) - 1.0) <= depth * 2.0 ** -23
        single = depth * 2.0 ** -22 * abs(theta)  # (FP32 sums in the operator itself, in both)
        out[basis] = theta
        attn.attn_heff_destroy(H)
        attn.attn_destroy(ctx)
    assert abs(out[1] - out[0]) <= single
