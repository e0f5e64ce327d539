"""The rotations of a disentangler update (u = -V W^T of Gamma = W sigma V^T by one-sided Jacobi)
where singular values of the environment nearly agree or lie far apart.

The tensors are pairs of neighbouring sites in (|00> + |11>) / sqrt(2), so that the density matrix
on two sites of different pairs is 1/4, and each disentangler has one term h = lambda - V s V^T with
max s = 2 lambda, whose shifted environment at u0 is Gamma = -u0^T V s V^T / 4: singular values s / 4 (and u = u0 the minimum).

Bounds: a column takes at most three rotations a sweep and about eight sweeps, each of unit
determinant to 2 roundings of FP64 (2^-53); 24 rotations adding up as a random walk give 1.1e-15,
1e-14 in the worst case of all in one direction. Tr(u Gamma) adds the rounding of 16 products,
below 2e-15 of the sum of the singular values."""
import numpy as np
import pytest

from inputs import normal
from oracle.tree import Tree
from tests.gpu_util import lib_and_ctx

pytestmark = pytest.mark.gpu

M = 4
CLOSE = [[1.0, 1.0 - g, 0.5, 0.3] for g in (1e-4, 1e-6, 1e-8, 1e-10, 1e-12)] + [
    [1.0, 1.0 - 1e-8, 1.0 - 2e-8, 1.0 - 3e-8], [1.0, 1.0, 0.5, 0.5], [1.0, 0.8, 0.8 + 1e-9, 0.8 + 3e-8]]
SPREAD = [[1.0, 0.5, 0.3, d] for d in (1e-4, 1e-6, 1e-8, 1e-10, 1e-12)] + [
    [1.0, 1e-4, 1e-8, 1e-12], [1.0, 1.0, 1e-6, 1e-12], [1.0, 0.7, 0.5, 0.3]]


def _orth(seed, k):
    q, r = np.linalg.qr(normal(seed, 700 + k, 16).reshape(4, 4))
    return q * np.sign(np.diag(r))


@pytest.mark.parametrize("spectra", [CLOSE, SPREAD], ids=["close", "spread"])
def test_update_stays_orthogonal(spectra):
    tree = Tree(16, M)
    raw = []
    for n, shape in enumerate(tree.shape):
        t = normal(5, n, int(np.prod(shape))).reshape(shape)
        t[:, :, 0] = 0.0  # the first state of a link: a pair below, the first state of both links above
        if shape[0] == 2:
            t[0, 0, 0] = t[1, 1, 0] = 1.0
        else:
            t[0, 0, 0] = 1.0
        raw.append(t)
    # the tensor that holds the norm: the first state of every link
    raw[tree.top_nodes()[0]][:] = 0.0
    raw[tree.top_nodes()[0]][0, 0, 0] = 1.0
    terms, us, hs = [], [], []
    for k, s in enumerate(spectra):
        v = _orth(1, k)
        lam = 0.5 * max(s)
        h = lam * np.eye(4) - v @ np.diag(s) @ v.T
        h = 0.5 * (h + h.T)
        terms.append(((k, 8 + k), h))
        hs.append((h, np.linalg.norm(h, 2)))
        us.append(_orth(2, k))
    attn, ctx = lib_and_ctx({"de_max_iter": 1})
    mod = attn.attn_model_terms(ctx, 16, terms)
    st = attn.attn_state_create(ctx, mod, M, raw)
    n = len(spectra)
    assert attn.attn_de_place(st, n) == n
    sites = attn.attn_de_sites(st, n)
    for k, u in enumerate(us):
        attn.attn_de_set(st, k, u)
    attn.attn_map_hamiltonian(st)
    env = []
    for k in range(n):
        assert sites[k] == (k, 8 + k)
        assert np.abs(attn.attn_rdm2(st, k) - 0.25 * np.eye(4)).max() <= 1e-14
        env.append(attn.attn_de_environment(st, k, us[k])[0])
        want = 0.25 * np.sort(spectra[k])[::-1]
        assert np.abs(np.linalg.svd(env[k], compute_uv=False) - want).max() <= 1e-14, k
    attn.attn_de_update(st)
    for k in range(n):
        u = attn.attn_de_get(st, k)
        assert np.abs(u.T @ u - np.eye(4)).max() <= 1e-14, (spectra[k], np.abs(u.T @ u - np.eye(4)).max())
        total = 0.25 * sum(spectra[k])
        assert abs(np.trace(u @ env[k]) + total) <= 1e-14 * total, spectra[k]
        attn.attn_de_set(st, k, u)  # accepts what it returned
    attn.attn_state_destroy(st)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)
