"""PC_VERDICT_FIRST with device outputs and no PC_MODE flag never waits for its
stream, whatever solver takes the call: behind other work on the stream the
call returns before that work ends, with the outputs of the single pass."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1401_2130_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    pc.build()
    pc.load()
    torch.cuda.init()


@pytest.mark.parametrize("W,L,p,n", [
    (64, 32, 0.9, 1),                       # dense: the streamed solver, one pass
    (132, 7, 0.13, 6), (132, 7, 0.3, 3),    # no window in shared memory: below and above the threshold
    (132, 7, 0.0, 2),                       # nothing percolates: nothing to select
    (8, 24, 0.2, 30), (40, 60, 0.17, 10),   # the wavefront solver
])
def test_call_returns_before_its_stream(W, L, p, n):
    import torch
    ref = pc.pc_inspect(W, L, p, 3, 2, n, mode=pc.PC_MODE_STREAM)
    bits = pc.pc_occupancy(W, L, p, 3, 2, n)
    calls = [lambda: pc.pc_inspect(W, L, p, 3, 2, n, verdict_first=True, device=True),
             lambda: pc.pc_inspect_occupancy(W, L, bits, mode=pc.PC_VERDICT_FIRST, device=True)]
    for call in calls:
        call()  # tables, pool
        torch.cuda.synchronize()
        early = False
        for _ in range(3):  # (the driver may wait when it grows its own memory for a graph)
            torch.cuda._sleep(int(6e8))  # about a third of a second
            done = torch.cuda.Event()
            done.record()
            g = call()
            early = early or not done.query()
            torch.cuda.synchronize()
        assert early
        for k in ("verdict", "first_hit", "m_stop", "mass"):
            assert np.array_equal(g[k].cpu().numpy(), ref[k]), k
        assert int(g["n_percolating"][0]) == ref["n_percolating"]
    h = pc.pc_inspect(W, L, p, 3, 2, n, verdict_first=True)  # host outputs read the error flags of both passes
    assert np.array_equal(h["mass"], ref["mass"])
