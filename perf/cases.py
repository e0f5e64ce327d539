"""Performance cases of libattn: what a user of the aTTN search has it do, through its public calls.

Families (``kind``):
  apply   one application of an explicit effective Hamiltonian, the call a caller's own Krylov solver makes
          at every step, in each of the four precisions (``attn_heff_create`` once, ``attn_heff_apply`` per pass)
  solve   one local eigenproblem from a start near its solution, as in every later sweep (``attn_eigsolve``)
  move    the isometry centre from the top of a tree to its last lowest tensor and back (``attn_move_centre``)
  build   a new disentangler layer taken into H': mapping, renormalisation of every link operator towards
          the centre, H_eff of the centre and its first application (``attn_map_hamiltonian``,
          ``attn_heff_build``, ``attn_heff_apply``)
  sweep   one aTTN sweep from random tensors (``attn_sweep``)
  update  one update of all disentanglers (``attn_de_update``)

Link dimensions and product counts are those of the TFIM lattices that the benchmark and the tests use: 4x4 with
m = 16, 8x8 with m = 32, 16x16 with m = 64, and the 32x32 top node with m = 128 and 288 products per link pair.
Tensors are normal deviates, link operators symmetric normal matrices of unit norm order, disentanglers random
orthogonal matrices.
"""
import math

import numpy as np
import torch

from paper_2507_21236_gb300 import attn

PAIR_P, PAIR_Q = (0, 0, 1), (1, 2, 2)  # slots of the pair kinds (0,1), (0,2), (1,2)
DTYPES = {"f64": 0, "f64_split": 0, "tf32": 2, "bf16": 3}  # attn_dtype; f64_split is a switch of the context


def listed():
    return [
        # the top node of a 4x4 lattice in the default precision: the smallest call, launches count
        dict(name="apply_f64_16", kind="apply", m0=16, m1=16, m2=16, n01=12, n02=12, n12=14, nt=0, dtype="f64"),
        # a heavy node of a 16x16 lattice, default precision (FP64 multiply-adds)
        dict(name="apply_f64_64", kind="apply", m0=64, m1=64, m2=64, n01=140, n02=140, n12=140, nt=0, dtype="f64"),
        # the 32x32 top node with the FP64 contractions as slice products: the matvec of its corrections
        dict(name="apply_split_128", kind="apply", m0=128, m1=128, m2=128, n01=288, n02=288, n12=288, nt=0,
             dtype="f64_split"),
        # a lower node of an 8x8 lattice, with products on all three links
        dict(name="apply_bf16_32", kind="apply", m0=32, m1=32, m2=32, n01=50, n02=45, n12=70, nt=12, dtype="bf16"),
        # a lower node of a 16x16 lattice, likewise, in the precision its sweeps use
        dict(name="apply_tf32_64", kind="apply", m0=64, m1=64, m2=64, n01=60, n02=61, n12=95, nt=24, dtype="tf32"),
        # the 32x32 top node: the headline matvec
        dict(name="apply_bf16_128", kind="apply", m0=128, m1=128, m2=128, n01=288, n02=288, n12=288, nt=0,
             dtype="bf16"),
        # a local solve of an 8x8 lattice with the default configuration
        dict(name="solve_f64_32", kind="solve", m0=32, m1=32, m2=32, n01=50, n02=45, n12=70, nt=12, dtype="f64",
             refine=0),
        # the local solve of the mixed policy at the 16x16, m = 128 size: TF32 Lanczos, FP64 corrections
        dict(name="solve_tf32_128", kind="solve", m0=128, m1=128, m2=128, n01=70, n02=70, n12=70, nt=0,
             dtype="tf32", refine=3),
        # the centre through a 16x16 tree: one QR and one small product per link
        dict(name="move_16x16_64", kind="move", L=16, m=64),
        # H_eff of the 16x16 top node under a new disentangler layer
        dict(name="build_16x16_64", kind="build", L=16, m=64, dtype="f64_split", compress=0, tri=0),
        # a whole sweep of a 4x4 lattice with the default configuration: many short calls, one after another
        dict(name="sweep_4x4_16", kind="sweep", L=4, m=16),
        # the disentangler update between two sweeps of an 8x8 lattice
        dict(name="update_8x8_32", kind="update", L=8, m=32),
    ]


def _log(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _products(rng, c, lo, hi, triples, budget):
    """Product counts within `budget` FLOPs."""
    for k in ("n01", "n02", "n12"):
        c[k] = _log(rng, lo, hi)
    c["nt"] = rng.choice((0, 0, _log(rng, 1, triples)))
    while _flops(c) > budget:
        for k in ("n01", "n02", "n12", "nt"):
            c[k] //= 2
    c["n01"] = max(c["n01"], 1)
    return c


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "apply", "solve", "move", "build", "sweep", "update"))
    if kind == "apply":
        dtype = rng.choice(("f64", "f64_split", "tf32", "bf16"))
        c = dict(kind=kind, dtype=dtype)
        for s in ("m0", "m1", "m2"):
            if dtype == "f64":
                c[s] = _log(rng, 4, 64)
            elif dtype == "f64_split":
                c[s] = _log(rng, 32, 128)
            else:  # the tensor-core tiles take multiples of 16
                c[s] = 16 * _log(rng, 1, 8)
        return _products(rng, c, 4, 288, 32, 2.5e10 if dtype == "f64" else 9e11)
    if kind == "solve":
        dtype = rng.choice(("f64", "tf32", "bf16"))
        c = dict(kind=kind, dtype=dtype, refine=0 if dtype == "f64" else 3)
        for s in ("m0", "m1", "m2"):
            c[s] = _log(rng, 8, 32) if dtype == "f64" else 16 * _log(rng, 2, 8)
        return _products(rng, c, 4, 70, 16, 1e9 if dtype == "f64" else 2e11)
    if kind == "move":
        return dict(kind=kind, L=rng.choice((4, 8, 16)), m=_log(rng, 6, 64))
    if kind == "build":
        L = rng.choice((4, 8, 16))
        return dict(kind=kind, L=L, m=_log(rng, 6, 64), dtype=rng.choice(("f64", "f64_split")),
                    compress=rng.choice((0, 1)), tri=rng.choice((0, 1)) if L < 16 else 0)
    if kind == "sweep":
        return dict(kind=kind, L=4, m=_log(rng, 6, 16))
    return dict(kind=kind, L=rng.choice((4, 8)), m=_log(rng, 6, 32))


# ------------------------------------------------------------------------------------------------ preparation
class Handles:
    """Library handles that are given back when the last reference goes (outputs that view a state's own
    buffers hold one)."""

    def __init__(self, **config):
        cfg = attn.attn_config_default()
        for k, v in config.items():
            setattr(cfg, k, v)
        self.ctx = attn.attn_create(cfg, torch.cuda.current_stream().cuda_stream or None)
        self.model = self.state = self.heff = None

    def __del__(self):
        if self.heff is not None:
            attn.attn_heff_destroy(self.heff)
        if self.state is not None:
            attn.attn_state_destroy(self.state)
        if self.model is not None:
            attn.attn_model_destroy(self.model)
        attn.attn_destroy(self.ctx)


class NodeView:
    """A node tensor in the library's own buffer, for torch.as_tensor."""

    def __init__(self, handles, node):
        self.handles = handles
        self.__cuda_array_interface__ = {
            "shape": attn.attn_node_shape(handles.state, node), "typestr": "<f8", "version": 3, "strides": None,
            "data": (attn.attn_node_device_ptr(handles.state, node), False)}


def _nodes(handles, nodes):
    return [torch.as_tensor(NodeView(handles, n), device="cuda") for n in nodes]


def _disentanglers(handles):
    return np.stack([attn.attn_de_get(handles.state, k) for k in range(handles.n_de)])


def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _operators(g, count, m, scale=1.0):
    a = _normal(g, count, m, m)
    return (a + a.transpose(1, 2)).mul_(0.5 * scale / math.sqrt(m))


def _heff_operators(c, g, solve):
    """Operators of an explicit H_eff: (internal operators, pairs, triples). For a solve the internal operators
    carry most of the energy and a gap, and the products couple the links weakly, as near a sweep's end;
    the start is the product of the internal operators' lowest vectors with some noise."""
    m = (c["m0"], c["m1"], c["m2"])
    n = (c["n01"], c["n02"], c["n12"])
    scale = 1.0 / math.sqrt(sum(n) + c["nt"]) if solve else 1.0
    hint = [_operators(g, 1, m[s])[0] for s in range(3)]
    start = _normal(g, *m)
    if solve:
        low = [torch.nn.functional.normalize(_normal(g, m[s]), dim=0) for s in range(3)]
        for s in range(3):
            hint[s] -= 4.0 * torch.outer(low[s], low[s])
        start *= 0.1 / start.norm()
        start += torch.einsum("a,b,c->abc", *low)
    pairs = {k: (_operators(g, n[k], m[PAIR_P[k]], scale), _operators(g, n[k], m[PAIR_Q[k]])) for k in range(3) if n[k]}
    triples = None
    if c["nt"]:
        triples = tuple(_operators(g, c["nt"], m[s], scale if s == 0 else 1.0) for s in range(3))
    return hint, pairs, triples, start


def _orthogonal(g):
    q, r = torch.linalg.qr(_normal(g, 4, 4))
    return (q * torch.sign(torch.diagonal(r))).cpu().numpy()


def _shapes(L, m):
    """Node shapes of the binary tree over L x L sites, layer by layer from the bottom."""
    out, layer, n = [], 1, L * L // 2
    dim = lambda e: min(2 ** (2 ** min(e, 10)), m)  # noqa: E731  the link above a layer-e node
    while n >= 2:
        out += [(dim(layer - 1), dim(layer - 1), dim(layer))] * n
        layer, n = layer + 1, n // 2
    return out


def _raw(c, g):
    """Random tensors of every node, on the host."""
    return [_normal(g, *s).cpu().numpy() for s in _shapes(c["L"], c["m"])]


def _tree(c, seed, **config):
    """A state with random tensors and random disentanglers."""
    g = _rng(seed)
    h = Handles(**config)
    if c.get("tri"):
        h.model = attn.attn_model_tri_heisenberg(h.ctx, c["L"], 1.0)
    else:
        h.model = attn.attn_model_tfim(h.ctx, c["L"], 3.0 if c["L"] == 4 else 3.04)
    h.state = attn.attn_state_create(h.ctx, h.model, c["m"], _raw(c, g))
    h.n_de = attn.attn_de_place(h.state, c["L"] * c["L"] // 4)
    for k in range(h.n_de):
        attn.attn_de_set(h.state, k, _orthogonal(g))
    attn.attn_map_hamiltonian(h.state)
    h.n_nodes, h.centre, _ = attn.attn_state_info(h.state)
    return h


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("apply", "solve"):
        config = dict(f64_split=int(c["dtype"] == "f64_split"))
        if kind == "solve":
            config = dict(matvec_dtype=DTYPES[c["dtype"]], refine_steps=c["refine"], f64_split=int(c["refine"] > 0))
        h = Handles(**config)
        hint, pairs, triples, x = _heff_operators(c, _rng(seed), kind == "solve")
        m = (c["m0"], c["m1"], c["m2"])
        h.heff = attn.attn_heff_create(h.ctx, m, hint, pairs, triples)
        torch.cuda.synchronize()
        return dict(kind=kind, handles=h, x=x, y=torch.empty_like(x), dtype=c["dtype"])
    if kind == "move":
        h = _tree(c, seed)
        return dict(kind=kind, handles=h, top=h.centre, target=c["L"] * c["L"] // 2 - 1,
                    path=_path(h.state, h.centre, c["L"] * c["L"] // 2 - 1))
    if kind == "build":
        h = _tree(c, seed, f64_split=int(c["dtype"] == "f64_split"), compress_terms=c["compress"])
        x = _normal(_rng(seed + 1), *attn.attn_node_shape(h.state, h.centre))
        return dict(kind=kind, handles=h, x=x, y=torch.empty_like(x))
    h = _tree(c, seed)
    return dict(kind=kind, handles=h, nodes=list(range(h.n_nodes)))


def _path(state, a, b):
    """Nodes between two tensors: up from b, and from a across the top link if b lies behind it."""
    def up(n):
        out = [n]
        while True:
            _, nb, back = attn.attn_node_neighbour(state, out[-1], 2)
            if back == 2:  # the other top tensor
                return out
            out.append(nb)
    below = up(b)
    return [a] + [n for n in reversed(below) if n != a]


# ------------------------------------------------------------------------------------------------------- a pass
def run(state):
    kind, h = state["kind"], state["handles"]
    if kind == "apply":
        attn.attn_heff_apply(h.heff, state["x"], state["y"], DTYPES[state["dtype"]])
        if state["dtype"] in ("tf32", "bf16"):
            # sums of BF16 or TF32 products in FP32: a caller keeps such vectors, and its Krylov basis, in FP32
            return state["y"].float()
        return state["y"]
    if kind == "solve":
        t = state["x"].clone()  # solved in place
        theta, _ = attn.attn_eigsolve(h.heff, t)
        # the FP64 corrections fix theta to FP64, and the vector to the square root of that
        return [theta, t if state["dtype"] == "f64" else t.float()]
    if kind == "move":
        attn.attn_move_centre(h.state, state["target"])
        attn.attn_move_centre(h.state, state["top"])
        return _nodes(h, state["path"])
    if kind == "build":
        attn.attn_map_hamiltonian(h.state)
        heff = attn.attn_heff_build(h.state, h.centre)
        attn.attn_heff_apply(heff, state["x"], state["y"], attn.ATTN_F64)
        attn.attn_heff_destroy(heff)
        return state["y"]
    if kind == "sweep":
        energy = attn.attn_sweep(h.state)
        return [energy, _nodes(h, state["nodes"]), _disentanglers(h)]
    change = attn.attn_de_update(h.state)
    return [change, attn.attn_de_energies(h.state, h.n_de), _disentanglers(h)]


# --------------------------------------------------------------------------------------------------------- work
def _flops(c):
    m = (c["m0"], c["m1"], c["m2"])
    V = m[0] * m[1] * m[2]
    f = 2.0 * sum(m) * V * (1 + c["nt"])
    for k, n in enumerate((c["n01"], c["n02"], c["n12"])):
        f += 2.0 * n * (m[PAIR_P[k]] + m[PAIR_Q[k]]) * V
    return f


def _operator_bytes(c):
    m = (c["m0"], c["m1"], c["m2"])
    b = 8.0 * (1 + c["nt"]) * sum(x * x for x in m)
    for k, n in enumerate((c["n01"], c["n02"], c["n12"])):
        b += 8.0 * n * (m[PAIR_P[k]] ** 2 + m[PAIR_Q[k]] ** 2)
    return b


def work(case):
    c, kind = case, case["kind"]
    if kind == "apply":
        V = c["m0"] * c["m1"] * c["m2"]
        return {"bytes": _operator_bytes(c) + 16.0 * V, "flops": _flops(c)}
    if kind == "solve":
        # 20 Lanczos steps; with corrections also 4 FP64 and up to 48 low-precision applications
        n = 20 + (c["refine"] * 17 + 1 if c["refine"] else 0)
        V = c["m0"] * c["m1"] * c["m2"]
        return {"bytes": _operator_bytes(c) + 16.0 * V, "flops": n * _flops(c) + 8.0 * 20 * 20 / 2 * V}
    shapes = _shapes(c["L"], c["m"])
    V = [a * b * d for a, b, d in shapes]
    if kind == "move":
        top, layers = len(shapes) - 1, int(math.log2(c["L"] * c["L"])) - 1
        path, n, width = [top], top, 2  # one node per layer and the other top tensor, each twice
        for _ in range(layers - 1):
            width *= 2
            n -= width
            path.append(n)
        f = sum(2 * (4.0 * V[i] * shapes[i][2] + 2.0 * V[i] * shapes[i][2]) for i in path) + 6.0 * V[top] * shapes[top][2]
        return {"bytes": 4 * 8.0 * (sum(V[i] for i in path) + V[top]), "flops": f}
    # products that cross the links of a node: on average about 1.5 per boundary site of its block, at each of
    # the two lower links; each is renormalised by two products with the node tensor
    f = b = 0.0
    layer, n, i = 1, c["L"] * c["L"] // 2, 0
    while n >= 2:
        crossing = 6.0 * math.sqrt(2.0 ** layer)
        f += n * crossing * 4.0 * shapes[i][2] * V[i]
        b += n * 8.0 * (V[i] + crossing * shapes[i][2] ** 2)
        i, layer, n = i + n, layer + 1, n // 2
    if kind == "sweep":
        return {"bytes": 2 * b, "flops": 22 * f}  # 20 Lanczos steps, the operators both ways
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------------------------------------------- exact
def _mode(x, s, a):
    """Operator a on slot s of x."""
    return torch.einsum(("ia,abc->ibc", "ib,abc->aic", "ic,abc->abi")[s], a, x)


def _apply_exact(hint, pairs, triples, x):
    y = sum(_mode(x, s, hint[s]) for s in range(3))
    for k, (a, b) in pairs.items():
        p, q = PAIR_P[k], PAIR_Q[k]
        for r in range(a.shape[0]):
            y += _mode(_mode(x, q, b[r]), p, a[r])
    if triples is not None:
        for r in range(triples[0].shape[0]):
            y += _mode(_mode(_mode(x, 2, triples[2][r]), 1, triples[1][r]), 0, triples[0][r])
    return y


def _lowest_exact(apply, x, steps=70):
    """Lowest eigenpair by Lanczos with full reorthogonalisation, run until it has converged."""
    basis, alpha, beta = [x / x.norm()], [], []
    for _ in range(steps):
        w = apply(basis[-1])
        alpha.append(float((w * basis[-1]).sum()))
        for _ in range(2):
            for v in basis:
                w -= (w * v).sum() * v
        b = float(w.norm())
        t = np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1)
        val, vec = np.linalg.eigh(t)
        if b * abs(vec[-1, 0]) < 1e-14 * abs(val[0]):
            break
        beta.append(b)
        basis.append(w / b)
    u = sum(float(z) * v for z, v in zip(vec[:, 0], basis))
    return float(val[0]), u * (torch.sign((u * x).sum()) / u.norm())


def _qr_exact(t, s):
    """Isometry and triangular factor of t with slot s as the columns, the factor's diagonal not negative."""
    a = t.movedim(s, 2)
    q, r = torch.linalg.qr(a.reshape(-1, a.shape[2]))
    sign = torch.where(torch.diagonal(r) < 0, -1.0, 1.0).to(t.dtype)
    return (q * sign).reshape(a.shape).movedim(2, s), r * sign[:, None]


def _move_exact(c, seed):
    g = _rng(seed)
    raw = [torch.as_tensor(t, device="cuda") for t in _raw(c, g)]
    top = len(raw) - 2  # the centre: the left top tensor
    chain, n, start, width = [top, top + 1], top + 1, top, 2  # down to the last lowest tensor
    while start > 0:
        width *= 2
        start -= width
        n = start + width - 1
        chain.append(n)
    tensors = {top: raw[top] / raw[top].norm()}
    for n in chain[1:]:
        tensors[n] = _qr_exact(raw[n], 2)[0]

    def hop(a, b, slot, back):
        tensors[a], r = _qr_exact(tensors[a], slot)
        tensors[b] = _mode(tensors[b], back, r)

    # the top tensors share their slot 2; further down the way goes through slot 1, the last child's
    slots = [(2, 2)] + [(1, 2)] * (len(chain) - 2)
    for (a, b), (s, t) in zip(zip(chain, chain[1:]), slots):
        hop(a, b, s, t)
    for (a, b), (s, t) in reversed(list(zip(zip(chain, chain[1:]), slots))):
        hop(b, a, t, s)
    return [tensors[n] for n in chain]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "apply":
        y = _apply_exact(*_heff_operators(c, _rng(seed), False))
        return y
    if kind == "solve":
        if _flops(c) > 1e11:
            return None  # 70 applications in 64 bits take too long
        hint, pairs, triples, x = _heff_operators(c, _rng(seed), True)
        theta, u = _lowest_exact(lambda v: _apply_exact(hint, pairs, triples, v), x)
        return [theta, u]
    if kind == "move":
        return _move_exact(c, seed)
    # a mapped Hamiltonian's renormalised operators, a sweep and an update have no short plain form
    return None
