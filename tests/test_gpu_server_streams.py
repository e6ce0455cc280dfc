"""A finished query's outputs do not wait for another query's run: a long query
first, then more short ones than it takes to go once round any small set of
streams.  And outputs of more than the pinned buffer holds."""
from __future__ import annotations

import time

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


def test_short_queries_behind_a_long_one():
    long_q = (8, 4000, 0.3, 1, 0, 12_000)
    short = [(W, L, p, 2, 0, 40) for W, L, p in [(4, 16, 0.2), (6, 9, 0.8), (16, 40, 0.18), (8, 24, 0.25)] * 10]
    srv = pc.Server(hbm_budget_bytes=2 << 30, max_slots=64, max_slots_per_query=16)
    try:
        want = {sp: pc.pc_inspect(*sp) for sp in set(short)}
        for sp in short[:4]:  # tables of each width
            assert srv.poll(srv.submit(sp), timeout_s=60.0) is not None
        first = srv.submit(long_q)
        t0 = time.time()
        while srv.poll(first, timeout_s=0.0) is None and time.time() - t0 < 0.02:
            pass  # it runs
        tickets = [srv.submit(sp) for sp in short]
        got = [srv.poll(t, timeout_s=60.0) for t in tickets]
        assert srv.poll(first, timeout_s=0.0) is None, "the short queries waited for the long one"
        for sp, g in zip(short, got):
            for k in KEYS:
                assert np.array_equal(g[k], want[sp][k]), (sp, k)
        big = srv.submit((2, 2, 0.3, 4, 0, 500_000))
        g = srv.poll(big, timeout_s=60.0)
        ref = pc.pc_inspect(2, 2, 0.3, 4, 0, 500_000)
        for k in KEYS:
            assert np.array_equal(g[k], ref[k]), k
        assert g["n_percolating"] == ref["n_percolating"]
        g = srv.poll(first, timeout_s=120.0)
        a = pc.pc_inspect(8, 4000, 0.3, 1, 0, 50)
        for k in KEYS:
            assert np.array_equal(g[k][:50], a[k]), k
    finally:
        srv.close()
