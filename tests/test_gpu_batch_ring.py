"""Block rings of a batch: a graph that is searched whole has room for some of
its root's children and queues the others as one frame, so the rings stay
small whatever the number of vertices."""
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


@pytest.mark.parametrize("n", [512, 1024, 2048, 4096])
def test_ring_bytes(ctx, n):
    import paper_1801_00202_gb300 as mce
    # as many alike graphs as keep every one of them whole on 2 and on 4 blocks
    graphs = [ctx.load_edges(n, synth.gnp(n, 4.0 / n, i)) for i in range(16)]
    used = []
    for blocks in (2, 4):
        base = ctx.mem_used()
        b = mce.Batch(ctx, graphs, mce.options(blocks=blocks))
        assert sum(x["split_graphs"] for x in b.buckets()) == 0
        used.append(ctx.mem_used() - base)
        b.close()
    frame = (8 + 2 * (n // 32)) * 4
    assert (used[1] - used[0]) / 2 <= 256 * (frame + 4) + 2048
    for g in graphs:
        g.free()


# more root children than the ring takes, one more, exactly as many
@pytest.mark.parametrize("pivot", ["greedy", "tx", "tomita"])
@pytest.mark.parametrize("kw", [dict(), dict(blocks=2, threads=64), dict(blocks=1, threads=32)], ids=["default", "2x64", "1x32"])
def test_rest_frame(ctx, pivot, kw):
    import paper_1801_00202_gb300 as mce
    star = lambda k: synth.join(synth.empty(1), 1, synth.empty(k), k)
    cases = [(1025, synth.gnp(1025, 0.02, 1)), (1025, synth.gnp(1025, 0.02, 2)), (2049, synth.gnp(2049, 0.005, 3)), (600, synth.gnp(600, 0.1, 4)),
             (700, synth.empty(700)), (96, synth.empty(96)), (97, synth.empty(97)), (98, synth.empty(98)),
             (1200, star(1199)), (300, synth.gnp(300, 0.3, 5))]
    graphs = [ctx.load_edges(n, uv) for n, uv in cases]
    for r, (n, uv) in zip(mce.enumerate_batch(ctx, graphs, mce.options(pivot=pivot, **kw)), cases):
        tree = oracle.ordered(n, uv, pivot)
        assert r["status"] == 0
        for k in ("count", "nodes", "internal", "dead_ends", "hash"):
            assert r[k] == tree[k], (n, k)
        assert np.array_equal(r["hist"], tree["hist"])
    for g in graphs:
        g.free()
