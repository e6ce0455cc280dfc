"""Outputs do not depend on the solver that a call takes.  The resident
solver's sum over the end layer has the order of the other solvers' (lane l of
one warp adds columns l, l + 32, .., then the lanes by halves), so a mass is
the same bits whichever of them ran, and with whatever CTA size."""
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


def _equal(a, b, what):
    for k in KEYS:
        assert np.array_equal(np.asarray(a[k]), np.asarray(b[k])), (what, k)


@pytest.mark.parametrize("W,L,p,n", [
    (0, 1, 0.5, 40), (0, 9, 0.95, 40),   # one column: one term
    (3, 1, 0.6, 200), (3, 2, 0.9, 200),  # 37 columns: a second round of five lanes
    (8, 12, 0.5, 300), (8, 40, 0.21, 300), (13, 1, 0.9, 50), (14, 14, 0.95, 60), (16, 16, 0.4, 60),
    (25, 1, 0.2, 300),                   # the most columns a CTA holds
])
def test_masses_of_the_solvers_are_the_same_bits(W, L, p, n):
    ref = pc.pc_inspect(W, L, p, 31, 7, n, mode=pc.PC_MODE_STREAM)
    assert ref["verdict"].any()
    for first in (False, True):
        _equal(pc.pc_inspect(W, L, p, 31, 7, n, mode=pc.PC_MODE_RESIDENT, verdict_first=first), ref, ("resident", first))
        _equal(pc.pc_inspect(W, L, p, 31, 7, n, verdict_first=first), ref, ("default", first))
