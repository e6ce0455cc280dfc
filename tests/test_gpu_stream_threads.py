"""Streamed, blocked and resident calls of different lattices from several
threads at once: each kernel's limit of dynamic shared memory is one for all
calls, so that none is refused for another's smaller one."""
from __future__ import annotations

import threading

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


def test_lattices_of_several_widths_at_once():
    import torch
    calls = [(W, L, dict(kw)) for W, L in [(3, 9), (12, 30), (30, 12), (64, 9)]
             for kw in ({"mode": pc.PC_MODE_STREAM}, {"mode": pc.PC_MODE_STREAM, "bits_only": True})]
    calls += [(2, 4, {"mode": pc.PC_MODE_RESIDENT}), (14, 14, {"mode": pc.PC_MODE_RESIDENT})]
    want = [pc.pc_inspect(W, L, 0.4, 1, 0, 6, **kw) for W, L, kw in calls]
    wrong = []

    def work(t):
        try:
            s = torch.cuda.Stream()
            for r in range(40):
                i = (3 * t + r) % len(calls)
                W, L, kw = calls[i]
                g = pc.pc_inspect(W, L, 0.4, 1, 0, 6, stream=s, **kw)
                for k in ("verdict", "first_hit", "m_stop", "mass"):
                    if not np.array_equal(g[k], want[i][k]):
                        wrong.append((calls[i], k))
        except Exception as e:  # the thread's, not the test's
            wrong.append(repr(e))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]
