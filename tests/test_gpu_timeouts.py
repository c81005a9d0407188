"""Very large wait budgets (callers' "no limit") end no search: ten times the
budget does not fit 64 bits, nor does its sum with the clock."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

BUDGETS = [2**64 - 1, 2**63 - 1, 2**64 // 10, 2**64 // 10 + 1]


@pytest.mark.parametrize("kw", [dict(blocks=1, threads=32), dict()], ids=["one-warp", "default"])
@pytest.mark.parametrize("n,p", [(90, 0.72), (150, 0.6)])
@pytest.mark.parametrize("budget", BUDGETS)
def test_no_limit(budget, n, p, kw):
    import paper_1801_00202_gb300 as mce
    mce.build()
    uv = synth.gnp(n, p, 3)
    tree = oracle.ordered(n, uv)
    with mce.Context(0) as ctx:
        g = ctx.load_edges(n, uv)
        opts = mce.options(timeout_ns=budget, **kw)
        for r in [g.enumerate(opts)] + mce.enumerate_batch(ctx, [g, g], opts) + [ctx.wait(ctx.submit(g, opts))]:
            for k in ("count", "nodes", "internal", "dead_ends", "hash"):
                assert r[k] == tree[k], k
            assert np.array_equal(r["hist"], tree["hist"])
