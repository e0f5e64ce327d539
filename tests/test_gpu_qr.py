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


def _clusters(M, k):
    """The clusters of eight CTAs that a matrix needs at least (256 rows and 200 KB each); over 19 it goes
    column by column."""
    rows = min(256, 200 * 1024 // 8 // (k | 1))
    return -(-M // (8 * rows)) if k <= 256 else 99


def _columns(kind, M, k, seed):
    a = normal(seed, 1, M * k).reshape(M, k)
    if kind == "dependent":  # 1e-9 beside a common direction
        a = a[:, :1] * normal(seed, 2, k) + 1e-9 * a
    elif kind == "repeated":
        a[:, 1::2] = a[:, 0:2 * (k // 2):2]
    elif kind == "ranges":  # sums that FP32 cannot hold, every third column nearly dependent
        a[:, 3::3] = a[:, :1] + 1e-7 * a[:, 3::3]
        a *= np.where(np.arange(k) % 2 == 0, 1e30, 1e-30)
    return a


# (160, 160, 160): 25600 rows of 160 columns are more than fits; the others take 2 to 14 clusters at least
@pytest.mark.parametrize("m", [61, 64, 100, 128, 160])
def test_moves_of_large_tensors(m):
    """8x8 lattice, from a top tensor [m, m, m] through each of its links and back, one QR after another
    on the same state: what is left behind is an isometry Q, the link's triangular factor R = Q^T T arrives
    in the neighbour, and Q R = T, for generic, dependent and repeated columns and columns outside FP32's
    range."""
    attn, ctx = lib_and_ctx()
    shapes = []
    for layer, n in enumerate((32, 16, 8, 4, 2)):
        cap = lambda e: min(2 ** (2 ** e), m)  # noqa: E731
        shapes += [(2 if layer == 0 else cap(layer),) * 2 + (cap(layer + 1),)] * n
    raw = [normal(5, n % 7, int(np.prod(s))).reshape(s) for n, s in enumerate(shapes)]
    assert (1 < _clusters(m * m, m) < 15) == (m < 160) and (_clusters(m * m, m) > 19) == (m == 160)
    mod = attn.attn_model_tfim(ctx, 8, 3.0)
    st = attn.attn_state_create(ctx, mod, m, raw)
    top = len(shapes) - 2
    eps = 2.0 ** -53
    for kind in ("generic", "dependent", "repeated", "ranges") if m < 160 else ("generic", "repeated"):
        for slot in (2, 0, 1):
            _, nb, back = attn.attn_node_neighbour(st, top, slot)
            cols = _columns(kind, m * m, m, 10 + slot)
            t = np.ascontiguousarray(np.moveaxis(cols.reshape(m, m, m), 2, slot))
            attn.attn_node_set(st, top, t)
            other = attn.attn_node_get(st, nb)
            attn.attn_move_centre(st, nb)
            q = np.moveaxis(attn.attn_node_get(st, top), slot, 2).reshape(m * m, m)
            assert np.abs(q.T @ q - np.eye(m)).max() < 1e-12, (kind, slot)
            r = q.T @ cols
            tol = 8 * m * eps * np.linalg.norm(cols, axis=0)  # (column by column: their scales differ)
            assert np.all(np.linalg.norm(q @ r - cols, axis=0) <= tol), (kind, slot)
            assert np.all(np.linalg.norm(np.tril(r, -1), axis=0) <= tol), (kind, slot)
            arrived = np.moveaxis(attn.attn_node_get(st, nb), back, 0).reshape(m, -1)
            o = np.moveaxis(other, back, 0).reshape(m, -1)
            sent = np.triu(r) @ o
            bound = ((tol + m * eps * np.linalg.norm(r, axis=0)) * np.linalg.norm(o, axis=1)).sum()
            assert np.linalg.norm(arrived - sent) <= bound, (kind, slot)
            attn.attn_move_centre(st, top)
            g = np.moveaxis(attn.attn_node_get(st, nb), back, 2).reshape(-1, m)
            assert np.abs(g.T @ g - np.eye(m)).max() < 1e-12, (kind, slot)
    attn.attn_state_destroy(st)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)
