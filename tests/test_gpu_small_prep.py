"""Graphs of up to 128 vertices, prepared by one launch: trees and results
against the oracle around every row width, wider input rows than needed, every
pivot rule; the order it leaves; and invalid rows, which queue nothing."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def run(n, rows, W, pivot):
    import torch
    import paper_1801_00202_gb300 as mce
    mce.build()
    o = mce.options(pivot=pivot)
    nb = mce.mce_scratch_bytes(n, o)
    sc = torch.empty(nb, dtype=torch.uint8, device="cuda")
    out = torch.full((mce.MCE_OUT_WORDS(n),), 77, dtype=torch.int64, device="cuda")
    d = torch.from_numpy(rows.view(np.int32).reshape(-1)).cuda()
    assert mce.mce_enumerate_device(n, W, d, o, sc, nb, out, torch.cuda.current_stream()) == mce.MCE_OK
    torch.cuda.synchronize()
    return mce, mce.decode_out(out, n)


@pytest.mark.parametrize("extra", [0, 5, 60])
@pytest.mark.parametrize("pivot", ["greedy", "tx", "nx", "tomita"])
@pytest.mark.parametrize("n,p", [(1, 0.5), (2, 1.0), (31, 0.5), (32, 0.6), (33, 0.6), (64, 0.5), (65, 0.5), (96, 0.4),
                                 (127, 0.3), (128, 0.3), (129, 0.3), (128, 0.0), (128, 1.0)])
def test_trees(n, p, pivot, extra):
    uv = synth.complete(n) if p == 1.0 else (synth.empty(n) if p == 0.0 else synth.gnp(n, p, 11 * n + 3))
    W = (n + 31) // 32 + extra
    mce, r = run(n, synth.to_bitset(n, uv, W), W, pivot)
    tree = oracle.ordered(n, uv, pivot)
    for k in ("count", "nodes", "internal", "dead_ends", "hash"):
        assert r[k] == tree[k], k
    assert np.array_equal(r["hist"], tree["hist"])


@pytest.mark.parametrize("n,word,bit", [(33, 0, 0), (33, 1, 1), (33, 1, 7), (64, 1, 31), (100, 3, 4)])
def test_invalid_rows(n, word, bit):
    uv = synth.gnp(n, 0.5, n)
    W = (n + 31) // 32
    rows = synth.to_bitset(n, uv, W).copy().reshape(n, W)
    rows[0, word] ^= np.uint32(1 << bit)  # the diagonal, a bit past n, or one direction of an edge
    mce, r = run(n, rows, W, "greedy")
    assert r["status"] == mce.MCE_EINVAL
