"""Runs of the warp tier long enough to fold their counters several times (a
structured core is one subproblem of 10^6 nodes and more)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivot", ["greedy", "tomita"])
@pytest.mark.parametrize("kw", [dict(blocks=1, threads=32), dict()], ids=["one-warp", "default"])
def test_folded_counters(kw, pivot):
    import paper_1801_00202_gb300 as mce
    mce.build()
    n, parts = 42, [synth.moon_moser(14)]
    for _ in range(4):  # cliques that make the average degree, and with it the sets, two words
        parts.append(synth.complete(40) + n)
        n += 40
    uv = np.concatenate(parts)
    tree = oracle.ordered(n, uv, pivot)
    with mce.Context(0) as ctx:
        r = ctx.load_edges(n, uv).enumerate(mce.options(pivot=pivot, **kw))
        for k in ("count", "nodes", "internal", "dead_ends", "hash"):
            assert r[k] == tree[k], k
        assert np.array_equal(r["hist"], tree["hist"])
