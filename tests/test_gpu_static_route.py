"""pc_inspect_static on both of its solvers: the resident one, on tables built
in the static array, and the wavefront one, at densities whose levels or start
layer overflow its queues.  Bits equal to the streamed solver's."""
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


@pytest.mark.parametrize("W,L,ps,n", [
    (0, 1, (0.5, 1.0), 700), (0, 40, (0.9,), 700), (1, 2, (0.3, 0.9), 3000), (4, 24, (0.2, 0.6, 0.95), 3000),
    (8, 16, (0.15, 0.25, 0.9), 2000), (12, 24, (0.18, 0.95), 400), (16, 16, (0.16, 0.5), 300),
    (20, 8, (0.3, 0.95), 200), (26, 1, (0.12, 0.9), 500),
])
def test_static_calls_at_every_density(W, L, ps, n):
    for p in ps:
        g = pc.pc_inspect_static(W, L, p, 5, 11, n)
        ref = pc.pc_inspect(W, L, p, 5, 11, n, mode=pc.PC_MODE_STREAM)
        for k in ("verdict", "first_hit", "m_stop", "mass"):
            assert np.array_equal(g[k], ref[k]), (p, k)
        assert g["n_percolating"] == ref["n_percolating"]
