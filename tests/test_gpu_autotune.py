"""The autotuner's candidates include what the library chooses by itself: a
batch of long searches, where no other block size comes near, keeps it."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_own_choice_is_a_candidate():
    import paper_1801_00202_gb300 as mce
    mce.build()
    with mce.Context(0) as ctx:
        cases = [(96, synth.gnp(96, 0.7, i)) for i in range(4)]
        graphs = [ctx.load_edges(n, uv) for n, uv in cases]
        own = mce.Batch(ctx, [graphs[i % 4] for i in range(160)])
        tuned = mce.Batch(ctx, [graphs[i % 4] for i in range(160)], mce.options(autotune=True))
        (a,), (b,) = own.buckets(), tuned.buckets()
        assert a["threads_per_block"] == 768 and b["tuned"] == 1
        assert b["threads_per_block"] == 768
        for batch in (own, tuned):
            for r, (n, uv) in zip(batch.run(), cases):
                tree = oracle.ordered(n, uv)
                for k in ("count", "nodes", "internal", "dead_ends", "hash"):
                    assert r[k] == tree[k], k
                assert np.array_equal(r["hist"], tree["hist"])


@pytest.mark.parametrize("pivot", ["greedy", "tx", "tomita"])
@pytest.mark.parametrize("n,p", [(96, 0.3), (300, 0.2), (1100, 0.05), (2100, 0.02)])
def test_both_register_bounds(n, p, pivot):
    # cheap graphs take 512 threads (one, two and four words a lane); a grid of
    # one block makes the same work long for its block
    import paper_1801_00202_gb300 as mce
    mce.build()
    with mce.Context(0) as ctx:
        cases = [(n, synth.gnp(n, p, i)) for i in range(3)]
        graphs = [ctx.load_edges(*c) for c in cases]
        count = 24
        for kw, threads in ((dict(), 512), (dict(blocks=1), None)):
            b = mce.Batch(ctx, [graphs[i % 3] for i in range(count)], mce.options(pivot=pivot, **kw))
            if threads:
                assert [x["threads_per_block"] for x in b.buckets()] == [threads]
            for r, (m, uv) in zip(b.run(), cases):
                tree = oracle.ordered(m, uv, pivot)
                for k in ("count", "nodes", "internal", "dead_ends", "hash"):
                    assert r[k] == tree[k], k
            b.close()
