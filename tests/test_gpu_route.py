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


@pytest.mark.parametrize("W,L,ps,n", [
    (8, 8, (0.45, 0.7), 4000), (14, 14, (0.2, 0.4, 0.95), 1), (3, 18, (0.15, 0.3), 20), (6, 2, (0.1, 0.3), 900),
    (20, 6, (0.6, 1.0), 500), (2, 5, (0.0, 1.0), 30), (25, 1, (0.15, 0.3), 700),
])
def test_default_calls_on_both_sides_of_the_line(W, L, ps, n):
    """pc_inspect without a mode: the densities lie on both sides of the one
    from which the resident solver takes the call."""
    import torch
    for p in ps:
        ref = pc.pc_inspect(W, L, p, 12, 3, n, mode=pc.PC_MODE_STREAM)
        g = pc.pc_inspect(W, L, p, 12, 3, n)
        _equal(g, ref, p)
        assert g["n_percolating"] == ref["n_percolating"]
        d = pc.pc_inspect(W, L, p, 12, 3, n, device=True, verdict_first=True)
        torch.cuda.synchronize()
        assert int(d.pop("n_percolating")[0]) == ref["n_percolating"]
        _equal({k: v.cpu().numpy() for k, v in d.items()}, ref, (p, "device"))
        b = pc.pc_inspect(W, L, p, 12, 3, n, bits_only=True)
        _equal(dict(b, mass=ref["mass"]), ref, (p, "verdicts"))
        assert not b["mass"].any()


@pytest.mark.parametrize("W,L,p,n", [(8, 48, 0.18, 100), (6, 36, 0.19, 200), (4, 48, 0.24, 700), (10, 40, 0.185, 16),
                                     (12, 24, 0.15, 100)])
def test_verdicts_first_below_the_threshold(W, L, p, n):
    """Levels of all configurations and then the masses of the few that
    percolate, where both would go in one pass without the flag."""
    g = pc.pc_inspect(W, L, p, 3, 0, n)
    _equal(pc.pc_inspect(W, L, p, 3, 0, n, verdict_first=True), g, "call")
    outs, _ = pc.pc_batch_run([(W, L, p, 3, 0, n), (W, L, p, 4, 0, n)], verdict_first=True)
    _equal(outs[0], g, "batch")


@pytest.mark.parametrize("W,L,p,n", [(16, 40, 0.4, 300), (20, 33, 0.95, 60), (24, 150, 0.6, 20), (30, 9, 0.8, 200)])
def test_dense_calls_in_one_pass(W, L, p, n):
    """Lattices beyond shared memory with large levels that nearly all
    percolate: levels and masses together, in planes of all layers (L <= 128)
    or in rings of them."""
    ref = pc.pc_inspect(W, L, p, 8, 1, n, mode=pc.PC_MODE_STREAM)
    assert ref["verdict"].all()
    _equal(pc.pc_inspect(W, L, p, 8, 1, n), ref, "call")
    outs, _ = pc.pc_batch_run([(W, L, p, 8, 1, n), (W, L, 0.0, 8, 1, 3), (W, L + 1, p, 8, 1, 2)])
    _equal(outs[0], ref, "batch")
    assert not outs[1]["verdict"].any() and not outs[1]["mass"].any()
