"""Link operators renormalised in one launch (tensors of up to 4096 entries) against the oracle's
sum of its per-product renormalised operators: dimensions that fill no block, the largest tensor
that takes the one-launch path, the first that does not (its one-sided products all go through the
tensor pair) and one whose links have lists on both sides of that rule."""
import numpy as np
import pytest

from oracle.de_update import build_problems, rdms
from tests.test_gpu_boundary import _close, _orth, _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,m,n_de", [(4, 3, 0), (4, 13, 4), (4, 16, 4), (8, 17, 16), (8, 33, 16)])
def test_internal_link_operators_match_oracle(L, m, n_de):
    attn, ctx, mod, st, ost, terms, tree, des, us = _pair(L, m, n_de)
    for node, slot in ((tree.top_nodes()[0], 0), (tree.top_nodes()[0], 2), (tree.node_id(2, 1), 1),
                       (tree.node_id(2, 0), 2)):
        kind, nb, back = tree.nbr[node][slot]
        n_open = attn.attn_renormalise(st, node, slot)
        ost.move_centre(nb)
        ops = ost.link_ops(nb, back)
        region = set(tree.region(nb, back))
        inner = [q for q in ops if set(ost.products[q][0]) <= region]
        ref = sum((ops[q] for q in inner), np.zeros((tree.shape[nb][back],) * 2))
        d, n2, has, h = attn.attn_link_operators(st, nb, back)
        assert n2 == n_open == len(ops) - len(inner)
        assert has == bool(inner)
        # FP64 on both sides, as the boundary tests have it
        assert np.abs(h - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())
        # the open operators act in H_eff of the node
        x = attn.attn_node_get(st, nb)
        H = attn.attn_heff_build(st, nb)
        y = attn.attn_heff_apply_host(H, x)
        want = ost.heff_apply(nb, x)
        assert np.abs(y - want).max() <= 1e-12 * np.abs(want).max()
        attn.attn_heff_destroy(H)
    _close(attn, ctx, mod, st)


@pytest.mark.parametrize("m", [17, 24])
def test_probe_lists_with_repeated_operators_match_oracle(m):
    """Density matrices and environments at link dimensions above the one-launch path, where the
    lists of probes open on two links repeat their operators; the boundary tests' bounds."""
    attn, ctx, mod, st, ost, terms, tree, des, us = _pair(8, m, 16)
    probs = build_problems(ost, terms, des)
    ref = rdms(ost, [tuple(d) for d in des])
    for k in range(len(des)):
        assert np.abs(attn.attn_rdm2(st, k) - ref[k]).max() <= 1e-12, k
        u = _orth(11, k)
        g, e = attn.attn_de_environment(st, k, u)
        gr, er = probs[k].gamma(u), probs[k].energy(u)
        assert np.abs(g - gr).max() <= 1e-12 * max(1.0, np.abs(gr).max()), k
        assert abs(e - er) <= 1e-12 * max(1.0, abs(er)), k
    attn.attn_de_update(st)  # all at once: the longest lists
    for p, u, e in zip(probs, us, attn.attn_de_energies(st, len(des))[:, 0]):
        assert abs(e - p.energy(u)) <= 1e-12 * max(1.0, abs(e))
    _close(attn, ctx, mod, st)
