"""A resumed FP64 run repeats the original's bits also where making the dense pair operators of an
H_eff barely pays (one application at a node of two pair kinds, a short Lanczos): the choice must
not depend on what the state did before it was saved."""
import numpy as np
import pytest

from inputs import raw_tree_tensors
from oracle.tree import Tree
from tests.gpu_util import lib_and_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [1, 2, 20])
@pytest.mark.parametrize("m,node", [(4, 0), (13, 0), (13, 3), (13, 9), (16, 5)])
def test_resumed_run_repeats_the_bits(tmp_path, m, node, depth):
    path = str(tmp_path / "state.bin")
    L = 4
    tree = Tree(L * L, m)
    raw = raw_tree_tensors(tree.shape, 3)
    attn, ctx = lib_and_ctx({"lanczos_depth": depth})
    mod = attn.attn_model_tfim(ctx, L, 3.0)
    st = attn.attn_state_create(ctx, mod, m, raw)
    attn.attn_de_place(st, 4)
    for _ in range(2):
        attn.attn_sweep(st)
    attn.attn_state_save(st, path)
    out = []
    st2 = attn.attn_state_create(ctx, mod, m, raw_tree_tensors(tree.shape, 5))
    attn.attn_state_load(st2, path)
    for s in (st, st2):
        attn.attn_move_centre(s, node)
        e = [attn.attn_energy(s)] + [attn.attn_sweep(s) for _ in range(2)]
        out.append((e, [attn.attn_node_get(s, i) for i in range(tree.n_nodes)]))
        attn.attn_state_destroy(s)
    attn.attn_model_destroy(mod)
    attn.attn_destroy(ctx)
    assert out[0][0] == out[1][0]
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))
