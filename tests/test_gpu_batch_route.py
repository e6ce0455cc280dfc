"""Batches whose queries go to different solvers: many small dense lattices
together on the resident one (each class of shared memory a launch), wide dense
ones together in one pool of slots, and sparse ones on the wavefront solver;
every query's outputs are pc_inspect's bits, and the reported threads those of
its launch."""
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


def _check(specs, **kw):
    import torch
    outs, res = pc.pc_batch_run(specs, **kw)
    d, _ = pc.pc_batch_run(specs, device=True, async_=True, **kw)
    torch.cuda.synchronize()
    for spec, o, r, dev in zip(specs, outs, res, d):
        if not spec[5]:
            continue
        ref = pc.pc_inspect(*spec, mode=pc.PC_MODE_STREAM)
        if kw.get("bits_only"):
            ref["mass"][:] = 0
        for k in KEYS:
            assert np.array_equal(o[k], ref[k]), (spec, k)
            assert np.array_equal(dev[k].cpu().numpy(), ref[k]), (spec, k, "device")
        assert r["n_percolating"] == ref["n_percolating"] == int(dev["n_percolating"][0])
    return res


DENSE = [(W, L, p, 40 + W, 3, n) for W, L, p, n in [
    (8, 70, 0.6, 40), (3, 5, 0.9, 300), (12, 20, 0.7, 30), (0, 1, 0.5, 100), (16, 16, 0.95, 20), (6, 6, 0.5, 0),
    (6, 9, 0.8, 200), (1, 3, 1.0, 10), (20, 8, 0.9, 5), (5, 4, 0.0, 60), (26, 1, 0.6, 33)]]


@pytest.mark.parametrize("kw", [{}, {"verdict_first": True}, {"bits_only": True}])
def test_small_dense_queries_together(kw):
    res = _check(DENSE, **kw)
    assert all(32 <= r["threads"] <= 640 for r, s in zip(res, DENSE) if s[5])


def test_wide_dense_queries_together():
    _check([(52, 20, 0.9, 1, 0, 3), (3, 9, 0.4, 6, 0, 50), (64, 12, 0.7, 2, 1, 2), (36, 30, 0.95, 3, 0, 4), (20, 60, 0.18, 4, 0, 20),
            (64, 20, 0.0, 5, 0, 2)])
    _check([(52, 20, 0.9, 1, 0, 3), (64, 12, 0.7, 2, 1, 2), (70, 12, 0.9, 3, 0, 2)], bits_only=True)


def test_sparse_and_dense_queries():
    _check([(8, 60, 0.2, 1, 0, 400), (4, 4, 0.9, 2, 0, 30), (14, 10, 0.16, 3, 0, 100), (30, 40, 0.5, 4, 0, 6)])


def test_outputs_beyond_the_pinned_buffer():
    """More than 4 MB of host outputs: each array goes straight to the caller's,
    and arrays that the caller leaves out are not touched."""
    specs = [(2, 2, 0.3, 1, 0, 300_000), (0, 1, 0.5, 2, 0, 7), (3, 2, 0.2, 3, 5, 200_000), (1, 1, 0.4, 4, 0, 0)]
    queries, outs = pc.batch_queries(specs, device=False)
    queries[2].first_hit = None
    queries[0].mass = None
    untouched = [outs[2]["first_hit"].copy(), outs[0]["mass"].copy()]
    _, res = pc.pc_batch_run(specs, outs=outs, queries=queries)
    assert np.array_equal(outs[2]["first_hit"], untouched[0]) and np.array_equal(outs[0]["mass"], untouched[1])
    for i, (spec, o, r) in enumerate(zip(specs[:3], outs, res)):
        ref = pc.pc_inspect(*spec)
        for k in KEYS:
            if (i, k) not in ((2, "first_hit"), (0, "mass")):
                assert np.array_equal(o[k], ref[k]), (spec, k)
        assert r["n_percolating"] == ref["n_percolating"]
