"""The warp tier at its edges, against the oracle's search tree: subproblems of
31 to 129 vertices around every set size, children counts around the largest
a frame's counter holds, whole graphs of 127 to 129 vertices, and stacks that
are paged out and given away."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1801_00202_gb300 as mce
    mce.build()
    c = mce.Context(0)
    yield c
    c.close()


def check(ctx, n, uv, pivot, repeat=1, **kw):
    import paper_1801_00202_gb300 as mce
    tree = oracle.ordered(n, uv, pivot)
    g = ctx.load_edges(n, uv)
    for _ in range(repeat):
        r = g.enumerate(mce.options(pivot=pivot, **kw))
        for k in ("count", "nodes", "internal", "dead_ends", "hash"):
            assert r[k] == tree[k], k
        assert np.array_equal(r["hist"], tree["hist"])
    g.free()


# (vertices of a clique, cliques): average degrees that make the search's sets
# one to four words
FILL = {1: (17, 6), 2: (40, 4), 3: (66, 4), 4: (100, 4)}


def core_graph(u, words):
    """Three vertices joined to a random graph of u vertices (children of the
    root with exactly u neighbours), and cliques beside it."""
    uv = synth.join(synth.empty(3), 3, synth.gnp(u, 0.35, u), u)
    n = u + 3
    m, k = FILL[words]
    parts = [uv]
    for _ in range(k):
        parts.append(synth.complete(m) + n)
        n += m
    return n, np.concatenate(parts)


@pytest.mark.parametrize("pivot", ["greedy", "tx", "nx", "tomita"])
@pytest.mark.parametrize("u", [31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129])
def test_subproblem_sizes(ctx, u, pivot):
    n, uv = core_graph(u, (u + 16) // 32)
    check(ctx, n, uv, pivot)


@pytest.mark.parametrize("pivot", ["greedy", "tomita"])
@pytest.mark.parametrize("n,uv", [
    (127, synth.gnp(127, 0.4, 1)), (128, synth.gnp(128, 0.4, 2)), (129, synth.gnp(129, 0.4, 3)),
    (128, synth.join(synth.empty(1), 1, synth.empty(127), 127)), (129, synth.join(synth.empty(1), 1, synth.empty(128), 128)),
    (130, synth.join(synth.empty(2), 2, synth.empty(128), 128)), (128, synth.empty(128)), (128, synth.complete(128)),
    (150, synth.complete(150))], ids=lambda a: str(a) if isinstance(a, int) else "")
def test_whole_graphs_and_stars(ctx, n, uv, pivot):
    check(ctx, n, uv, pivot)


@pytest.mark.parametrize("kw", [dict(), dict(blocks=1, threads=32), dict(blocks=2, threads=512), dict(blocks=40, threads=64)],
                         ids=["default", "1x32", "2x512", "40x64"])
@pytest.mark.parametrize("n,uv,pivot", [(36, synth.moon_moser(12), "greedy"), (90, synth.gnp(90, 0.72, 4), "nx"),
                                        (136, synth.gnp(136, 0.6, 5), "greedy"), (150, synth.gnp(150, 0.5, 6), "tomita")],
                         ids=["mm36", "gnp90", "gnp136", "gnp150"])
def test_paged_and_given_frames(ctx, n, uv, pivot, kw):
    check(ctx, n, uv, pivot, repeat=1 if kw.get("blocks") == 1 else 4, **kw)
