"""Centre moves (one QR per link) at the shapes where the one-launch QR changes its split: one
cluster or several, rows that do not divide, single columns, square and dependent columns. The
tensors left behind are isometries and the state does not change (its tensors contract to the
same two-node tensor)."""
import numpy as np
import pytest

from inputs.synth import normal
from tests.gpu_util import lib_and_ctx

pytestmark = pytest.mark.gpu


def _shapes(m):
    cap = lambda e: min(2 ** (2 ** e), m)  # noqa: E731
    return [(2, 2, cap(1))] * 8 + [(cap(1), cap(1), cap(2))] * 4 + [(cap(2), cap(2), cap(3))] * 2


@pytest.mark.parametrize("m", [2, 4, 7, 13, 16, 33, 64, 100, 128])
@pytest.mark.parametrize("scale", [1.0, 1e-9])
def test_move_keeps_the_state_and_leaves_isometries(m, scale):
    """4x4 lattice; the top tensors have one link of dimension m (up to 256 at 128 columns).
    `scale` shrinks all but the first columns' new directions: strongly dependent columns, as a
    converged state has them, where a single Gram-Schmidt pass loses orthogonality."""
    attn, ctx = lib_and_ctx()
    shapes = _shapes(m)
    raw = [normal(5, n, int(np.prod(s))).reshape(s) for n, s in enumerate(shapes)]
    mod = attn.attn_model_tfim(ctx, 4, 3.0)
    st = attn.attn_state_create(ctx, mod, m, raw)
    top, other = len(shapes) - 2, len(shapes) - 1
    t = attn.attn_node_get(st, top)
    k = shapes[top][2]
    base = t[:, :, :1] * normal(7, 1, k)[None, None, :]
    t = base + scale * t
    attn.attn_node_set(st, top, t)
    before = np.einsum("abk,cdk->abcd", t, attn.attn_node_get(st, other))
    attn.attn_move_centre(st, other)
    q, c = attn.attn_node_get(st, top), attn.attn_node_get(st, other)
    g = np.einsum("abk,abl->kl", q, q)
    assert np.abs(g - np.eye(k)).max() < 1e-12
    after = np.einsum("abk,cdk->abcd", q, c)
    # backward error of a QR: a small multiple of k roundings of the tensor's norm
    assert np.linalg.norm(after - before) <= 8 * k * 2.0 ** -53 * np.linalg.norm(before)
    attn.attn_state_destroy(st)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)


def test_dependent_columns_are_completed():
    """Exactly repeated columns: their R diagonal is zero, the tensor left behind is an isometry
    all the same, and the state is kept."""
    attn, ctx = lib_and_ctx()
    m = 16
    shapes = _shapes(m)
    raw = [normal(6, n, int(np.prod(s))).reshape(s) for n, s in enumerate(shapes)]
    mod = attn.attn_model_tfim(ctx, 4, 3.0)
    st = attn.attn_state_create(ctx, mod, m, raw)
    top, other = len(shapes) - 2, len(shapes) - 1
    t = np.zeros(shapes[top])
    for c in range(m):  # unit vectors, each twice
        t[c // 2, 0, c] = 1.0 + c // 2
    attn.attn_node_set(st, top, t)
    before = np.einsum("abk,cdk->abcd", t, attn.attn_node_get(st, other))
    attn.attn_move_centre(st, other)
    q, c = attn.attn_node_get(st, top), attn.attn_node_get(st, other)
    assert np.abs(np.einsum("abk,abl->kl", q, q) - np.eye(m)).max() < 1e-12
    assert np.abs(np.einsum("abk,cdk->abcd", q, c) - before).max() < 1e-13 * np.abs(before).max()
    attn.attn_state_destroy(st)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)


@pytest.mark.parametrize("even, odd", [(1e40, 1e40), (1e-40, 1e-40), (1e30, 1e-30), (1.0, 1e60)])
def test_columns_outside_the_range_of_fp32(even, odd):
    """Columns whose sums, or products of sums, FP32 cannot hold (the one-launch QR takes small corrections
    in FP32); some of them nearly dependent, so that both Gram-Schmidt passes count."""
    attn, ctx = lib_and_ctx()
    m = 33
    shapes = _shapes(m)
    raw = [normal(8, n, int(np.prod(s))).reshape(s) for n, s in enumerate(shapes)]
    mod = attn.attn_model_tfim(ctx, 4, 3.0)
    st = attn.attn_state_create(ctx, mod, m, raw)
    top, other = len(shapes) - 2, len(shapes) - 1
    t = attn.attn_node_get(st, top)
    t[:, :, 3::3] = t[:, :, :1] + 1e-7 * t[:, :, 3::3]
    k = shapes[top][2]
    t = t * np.where(np.arange(k) % 2 == 0, even, odd)[None, None, :]
    attn.attn_node_set(st, top, t)
    o = attn.attn_node_get(st, other)
    before = np.einsum("abk,cdk->abcd", t, o)
    attn.attn_move_centre(st, other)
    q, c = attn.attn_node_get(st, top), attn.attn_node_get(st, other)
    assert np.abs(np.einsum("abk,abl->kl", q, q) - np.eye(k)).max() < 1e-12
    after = np.einsum("abk,cdk->abcd", q, c)
    # backward error of a QR: a small multiple of k roundings of the tensor's norm
    assert np.linalg.norm(after - before) <= 8 * k * 2.0 ** -53 * np.linalg.norm(before)
    attn.attn_state_destroy(st)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)
