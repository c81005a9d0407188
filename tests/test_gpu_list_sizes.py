"""A listing call without room for an offset: the sizes of the listing, from
the counting search, for every pivot rule and around a set's word sizes."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flag", ["MCE_LIST", "MCE_LIST_SORTED"])
@pytest.mark.parametrize("n,p,pivot", [(0, 0.0, "greedy"), (1, 0.0, "greedy"), (33, 0.6, "tx"), (128, 0.4, "nx"),
                                       (129, 0.4, "tomita"), (300, 0.2, "greedy"), (1100, 0.05, "greedy")])
def test_sizes_of_a_listing(n, p, pivot, flag):
    import paper_1801_00202_gb300 as mce
    mce.build()
    ctx = mce.Context(0)
    uv = synth.gnp(n, p, n + 5) if n > 1 else synth.empty(n)
    g = ctx.load_edges(n, uv)
    o = mce.options(pivot=pivot, flags=getattr(mce, flag))
    r = g.enumerate(o, raise_on_error=False, list_cap=0, off_cap=0)
    tree = oracle.ordered(n, uv, pivot)
    assert r["rc"] == mce.MCE_ETRUNC
    for k in ("count", "nodes", "internal", "dead_ends", "hash"):
        assert r[k] == tree[k], k
    hist = np.asarray(tree["hist"], dtype=np.uint64)
    assert np.array_equal(r["hist"], hist)
    assert r["list_ids_needed"] == int((hist * np.arange(hist.size, dtype=np.uint64)).sum())
    full = g.enumerate(o, list_cap=r["list_ids_needed"], off_cap=r["count"] + 1)
    assert full["rc"] == 0 and full["list_off"][-1] == r["list_ids_needed"]
    g.free()
    ctx.close()
