"""The degeneracy order of the outer loop, through the search trees that it
fixes (the oracle's, node for node), where its lists and minima change shape:
vertices around a chunk of 32 and a super-chunk of 1,024, lists of up to and
over 128 neighbours, averages below and above 128, equal degrees throughout and isolated vertices."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

GRAPHS = [(n, p, synth.gnp(n, p, 3 * n + 1)) for n, p in
          [(2, 1.0), (31, 0.5), (32, 0.5), (33, 0.5), (180, 0.45), (290, 0.42), (330, 0.4), (1023, 0.02), (1024, 0.02), (1025, 0.02),
           (2050, 0.01), (4500, 0.002)]]
GRAPHS += [(1500, "cycle", synth.cycle(1500)), (400, "star", synth.join(synth.empty(1), 1, synth.empty(399), 399)),
           (700, "isolated", synth.gnp(300, 0.2, 9)), (131, "complete", synth.complete(131))]


@pytest.mark.parametrize("n,what,uv", GRAPHS, ids=[f"{n}-{w}" for n, w, _ in GRAPHS])
def test_outer_trees(n, what, uv):
    import paper_1801_00202_gb300 as mce
    mce.build()
    ctx = mce.Context(0)
    g = ctx.load_edges(n, uv)
    r = g.enumerate(mce.options(flags=mce.MCE_OUTER))
    tree = oracle.outer(n, uv)
    for k in ("count", "nodes", "internal", "dead_ends", "hash"):
        assert r[k] == tree[k], k
    g.free()
    ctx.close()
