"""Root frames of batched graphs against the oracle's tree: frames of several
children in whole graphs and in parts, every set size of the warp tier, dense
graphs, and children counts around the largest that a frame's counter holds
(127), which a batch takes into the tier with 128-vertex sets."""
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


def check(ctx, cases, pivot, **kw):
    import paper_1801_00202_gb300 as mce
    graphs = [ctx.load_edges(n, uv) for n, uv in cases]
    b = mce.Batch(ctx, graphs, mce.options(pivot=pivot, **kw))
    split = sum(x["split_graphs"] for x in b.buckets())
    for _ in range(2):
        for r, (n, uv) in zip(b.run(), cases):
            tree = oracle.ordered(n, uv, pivot)
            assert r["status"] == 0
            for k in ("count", "nodes", "internal", "dead_ends", "hash"):
                assert r[k] == tree[k], (n, k)
            assert np.array_equal(r["hist"], tree["hist"])
    b.close()
    for g in graphs:
        g.free()
    return split


def star(hubs, leaves):
    return hubs + leaves, synth.join(synth.empty(hubs), hubs, synth.empty(leaves), leaves)


def core(u):
    """Three vertices joined to a random graph of u vertices, and four cliques."""
    uv, n = [synth.join(synth.empty(3), 3, synth.gnp(u, 0.35, u), u)], u + 3
    for _ in range(4):
        uv.append(synth.complete(100) + n)
        n += 100
    return n, np.concatenate(uv)


@pytest.mark.parametrize("pivot", ["greedy", "tomita"])
def test_children_counts(ctx, pivot):
    check(ctx, [star(1, 127), star(1, 128), star(1, 129), star(2, 128), star(2, 127)] + [core(u) for u in (127, 128, 129)], pivot)


@pytest.mark.parametrize("pivot", ["greedy", "tx", "tomita"])
@pytest.mark.parametrize("n,p", [(129, 0.05), (160, 0.1), (220, 0.1), (300, 0.2), (420, 0.12), (1100, 0.02), (1100, 0.07)])
def test_whole_graphs(ctx, n, p, pivot):
    # as many as keep every graph whole on 4 blocks
    assert check(ctx, [(n, synth.gnp(n, p, i)) for i in range(17)], pivot, blocks=4) == 0


@pytest.mark.parametrize("kw", [dict(blocks=2, threads=64), dict(blocks=3, threads=512), dict()], ids=["2x64", "3x512", "default"])
@pytest.mark.parametrize("n,p", [(700, 0.06), (1500, 0.02), (2500, 0.02)])
def test_parts(ctx, n, p, kw):
    assert check(ctx, [(n, synth.gnp(n, p, i)) for i in range(3)], "greedy", **kw) == 3


@pytest.mark.parametrize("pivot", ["greedy", "nx"])
def test_dense_graphs(ctx, pivot):
    check(ctx, [(48, synth.gnp(48, 0.8, 1)), (64, synth.gnp(64, 0.75, 2)), (33, synth.moon_moser(11)), (50, synth.gnp(50, 0.9, 3)),
                (131, synth.gnp(131, 0.7, 4)), (150, synth.complete(150))] * 3, pivot)
