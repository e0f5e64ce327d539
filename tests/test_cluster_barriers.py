"""Kernels that use distributed shared memory, read as text (a missing barrier may fault a GPU, so no
kernel runs for this): a CTA's shared memory exists for the others of its cluster from the first
cluster barrier, which shows that every CTA has started, until the last one, before which none may leave."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_21236_gb300", "csrc")


def _functions(text):
    """(head, body) of every top-level function of a source text without comments."""
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    out = []
    for m in re.finditer(r"^(?:template <[^\n]*>\n)?(?:static )?(?:__global__|__device__)[^;{]*\{", text, flags=re.M):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out.append((m.group(0), text[m.end():i - 1]))
    return out


FUNCTIONS = [(os.path.basename(p), h, b) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
             for h, b in _functions(open(p).read())]
REMOTE = [f for f in FUNCTIONS if "map_shared_rank" in f[2]]
NAME = re.compile(r"(\w+)\(")


def _name(head):
    return [n for n in NAME.findall(head) if n not in ("__launch_bounds__", "sizeof")][0]


def test_cluster_kernels_are_found():
    assert {_name(h) for _, h, _ in REMOTE} == {"lz_tail_kernel", "qr_reduce"}


@pytest.mark.parametrize("file,head,body", REMOTE, ids=[_name(h) for _, h, _ in REMOTE])
def test_barrier_before_the_first_remote_access(file, head, body):
    assert ".sync()" in body[:body.index("map_shared_rank")], file


@pytest.mark.parametrize("name", ["lz_tail_kernel", "qr_slab_kernel"])
def test_barrier_before_a_cta_leaves(name):
    """The kernel ends with a cluster barrier, and so does every early return after its first one."""
    body = [b for _, h, b in FUNCTIONS if _name(h) == name][0]
    barrier = r"(?:cl|cg::this_cluster\(\))\.sync\(\);"
    assert re.search(barrier + r"\s*$", body)
    first = re.search(barrier, body).end()
    for m in re.finditer(r"\breturn;", body[first:]):
        assert re.search(barrier + r"\s*$", body[first:first + m.start()])
