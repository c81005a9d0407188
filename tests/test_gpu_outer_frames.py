"""Outer-loop subproblems of more than 128 vertices, which start from frames
of their root's children (P, X and R carried in), against the definition's
results and a search of the graph as one."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivot", ["greedy", "tx", "tomita"])
@pytest.mark.parametrize("n,p", [(600, 0.3), (1200, 0.15), (2200, 0.09)])
@pytest.mark.parametrize("kw", [dict(), dict(threads=32), dict(threads=512)], ids=["default", "32", "512"])
def test_large_subproblems(n, p, pivot, kw):
    import paper_1801_00202_gb300 as mce
    mce.build()
    uv = synth.gnp(n, p, 7)
    with mce.Context(0) as ctx:
        g = ctx.load_edges(n, uv)
        ref = oracle.tomita(n, uv)
        a, b = g.enumerate(mce.options(pivot=pivot, outer=True, **kw)), g.enumerate(mce.options(pivot=pivot))
        for r in (a, b):
            assert r["count"] == ref["count"] and r["hash"] == ref["hash"]
            assert np.array_equal(r["hist"], ref["hist"])
        # the outer loop's tree does not depend on how a block searches it
        c = g.enumerate(mce.options(pivot=pivot, outer=True, threads=64))
        for k in ("nodes", "internal", "dead_ends"):
            assert a[k] == c[k], k
