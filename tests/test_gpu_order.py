"""The maximum-degree-first order kernel against the oracle's order, vertex for
vertex, at the sizes where its rounds change shape: below and above 128
candidates and the 512- and 1,024-thread blocks, rows in shared memory and in
L2, whole degree classes and a class of more than 128 vertices (regular
graphs), and row strides wider than needed."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

GRAPHS = [(n, p, synth.gnp(n, p, 7 * n + 1)) for n, p in
          [(1, 0.5), (2, 0.5), (33, 0.6), (127, 0.5), (128, 0.4), (129, 0.5), (300, 0.05), (512, 0.8), (513, 0.3),
           (1024, 0.3), (1025, 0.1), (2049, 0.03), (4096, 0.01)]]
GRAPHS += [(129, "empty", synth.empty(129)), (500, "complete", synth.complete(500)), (1000, "cycle", synth.cycle(1000)),
           (180, "moon_moser", synth.moon_moser(60)), (4096, "cycle", synth.cycle(4096)),
           (300, "multipartite", synth.complete_multipartite([150, 100, 50])),
           (400, "star", synth.join(synth.empty(1), 1, synth.empty(399), 399))]


@pytest.mark.parametrize("extra", [0, 3])
@pytest.mark.parametrize("n,what,uv", GRAPHS, ids=[f"{n}-{w}" for n, w, _ in GRAPHS])
def test_order_matches_oracle(n, what, uv, extra):
    import torch
    import paper_1801_00202_gb300 as mce
    mce.build()
    W = (n + 31) // 32 + extra
    rows = torch.from_numpy(synth.to_bitset(n, uv, W).view(np.int32).reshape(-1)).cuda()
    order = torch.zeros(n, dtype=torch.int32, device="cuda")
    assert mce.mce_order(n, W, rows, order, torch.cuda.current_stream()) == mce.MCE_OK
    torch.cuda.synchronize()
    assert np.array_equal(order.cpu().numpy(), oracle.mdf_order(n, uv))
