"""Calls with little device memory left: rows drawn ahead need every
configuration's maps at once, and where these cannot be had the groups draw
their own rows, fewer of them at a time."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1401_2130_gb300 as pc

pytestmark = pytest.mark.gpu

KEYS = ("verdict", "first_hit", "m_stop", "mass")


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    pc.build()
    pc.load()
    torch.cuda.init()


def test_rows_drawn_ahead_without_their_memory():
    import torch
    W, L, p, n = 64, 2048, 0.16, 140
    ref = pc.pc_inspect(W, L, p, 5, 0, n)
    bits = pc.pc_inspect(W, L, p, 5, 0, n, bits_only=True)
    maps = 12 * pc.pc_lattice_layout(W)["P"] * ((L + 31) // 32) * n
    torch.cuda.synchronize()
    pc.load().pc_shutdown()  # the scratch pool's memory goes back
    torch.cuda.empty_cache()
    left = 500 << 20
    assert left < maps < 2 << 30
    hog = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        g = pc.pc_inspect(W, L, p, 5, 0, n)
        b = pc.pc_inspect(W, L, p, 5, 0, n, bits_only=True)
    finally:
        del hog
        torch.cuda.empty_cache()
    for k in KEYS:
        assert np.array_equal(g[k], ref[k]), k
        assert np.array_equal(b[k], bits[k]), k
