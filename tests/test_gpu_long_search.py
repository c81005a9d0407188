"""Both register bounds of the single-graph search, which the number of
expected maximal cliques chooses between: very dense graphs of few cliques
(expected to be long, so they take the 768-thread blocks) and the same with
512-thread blocks asked for, against the oracle's tree."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def almost_complete(n, pairs):
    """The complete graph without `pairs` disjoint edges: 2^pairs cliques."""
    uv = synth.complete(n)
    gone = (uv[:, 0] // 2 == uv[:, 1] // 2) & (uv[:, 0] < 2 * pairs)
    return uv[~gone]


@pytest.mark.parametrize("threads", [0, 32, 512])
@pytest.mark.parametrize("pivot", ["greedy", "tx", "tomita"])
@pytest.mark.parametrize("n,pairs", [(128, 13), (129, 13), (300, 10), (300, 0), (1100, 6)])
def test_trees(n, pairs, pivot, threads):
    import paper_1801_00202_gb300 as mce
    mce.build()
    ctx = mce.Context(0)
    uv = almost_complete(n, pairs)
    g = ctx.load_edges(n, uv)
    r = g.enumerate(mce.options(pivot=pivot, **({"threads": threads} if threads else {})))
    tree = oracle.ordered(n, uv, pivot)
    for k in ("count", "nodes", "internal", "dead_ends", "hash"):
        assert r[k] == tree[k], k
    assert np.array_equal(r["hist"], tree["hist"])
    g.free()
    ctx.close()
