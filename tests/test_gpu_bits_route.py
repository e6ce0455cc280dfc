"""Caller occupancies at every density: a sample on the device chooses the
launches that run, so each choice, and calls that mix densities, must give the
streamed solver's bits.  Sizes on both sides of each rule: start layers that
overflow tables sized for few sites, lattices beyond shared memory, and wide
ones that the whole device works on where they are dense."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_1401_2130_gb300 as pc

pytestmark = pytest.mark.gpu

KEYS = ("verdict", "first_hit", "m_stop", "mass")


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    pc.build()
    pc.load()
    torch.cuda.init()


def _bits(W, L, ps, n):
    """n configurations of each density of ps, in turn."""
    import torch
    parts = [pc.pc_occupancy(W, L, p, 40 + k, 0, n) for k, p in enumerate(ps)]
    return torch.stack(parts, 1).reshape(n * len(ps), -1).contiguous()


def _check(W, L, bits, what):
    import torch
    n = bits.shape[0]
    ref = pc.pc_inspect_occupancy(W, L, bits, mode=pc.PC_MODE_STREAM)
    for mode in (0, pc.PC_BITS_ONLY, pc.PC_VERDICT_FIRST):
        # the sample comes in time, or behind other work on the stream it does not
        for device, busy in ((False, False), (True, False), (True, True), (False, True)):
            if busy:
                torch.cuda._sleep(1_000_000)
            g = pc.pc_inspect_occupancy(W, L, bits, mode=mode, device=device)
            torch.cuda.synchronize()
            g = {k: v.cpu().numpy() if hasattr(v, "cpu") else v for k, v in g.items()}
            for k in KEYS:
                want = np.zeros(n, np.float32) if k == "mass" and mode == pc.PC_BITS_ONLY else ref[k]
                assert np.array_equal(g[k], want), (what, mode, device, busy, k)
            assert int(np.asarray(g["n_percolating"]).reshape(-1)[0]) == ref["n_percolating"]


@pytest.mark.parametrize("W,L,n", [
    (0, 3, 40), (2, 7, 50), (8, 48, 16), (8, 16, 200), (7, 90, 30), (12, 24, 60), (16, 5, 150), (26, 1, 100),
    (14, 60, 40), (30, 60, 8), (20, 150, 10),     # beyond shared memory: rings or planes
])
def test_every_density(W, L, n):
    for ps in ((0.0,), (0.17,), (0.24, 0.26), (0.5,), (0.95,), (1.0,), (0.05, 0.9), (0.1, 0.2, 0.4, 0.8)):
        _check(W, L, _bits(W, L, ps, n), ps)


@pytest.mark.parametrize("W,L,n", [(64, 12, 2), (40, 40, 3), (64, 33, 1), (36, 130, 2), (130, 5, 2)])
def test_wide_lattices(W, L, n):
    for ps in ((0.15,), (0.3,), (0.6,), (0.97,), (0.1, 0.9)):
        _check(W, L, _bits(W, L, ps, n), ps)


def test_one_dense_configuration_among_sparse_ones():
    W, L, n = 10, 30, 300
    bits = _bits(W, L, (0.12,), n)
    bits[211] = _bits(W, L, (0.97,), 1)[0]
    _check(W, L, bits, "one dense")
    occ = np.zeros((4, (3 * W * (W + 1) + 1) * L), np.uint8)
    occ[1], occ[2, ::2] = 1, 1
    import torch
    full = torch.from_numpy(oracle.pack_bits(occ).view(np.int32)).cuda()
    ref = oracle.inspect(W, L, occ=occ, mode="markov", threads=4)
    g = pc.pc_inspect_occupancy(W, L, full)
    for k in ("verdict", "first_hit", "m_stop"):
        assert np.array_equal(g[k].astype(np.int64), np.asarray(ref[k]).astype(np.int64)), k


@pytest.mark.parametrize("W,L,p", [(8, 24, 0.2), (8, 24, 0.8), (40, 70, 0.2), (40, 70, 0.8)])
def test_captured_calls(W, L, p):
    """Device outputs under stream capture: nothing waits for the sample."""
    import torch
    bits = _bits(W, L, (p,), 5)
    ref = pc.pc_inspect_occupancy(W, L, bits)
    out = pc._alloc_outputs(5, True, pc.ALL_OUTPUTS)
    pc.pc_inspect_occupancy(W, L, bits, device=True, out=out)  # tables of W
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        pc.pc_inspect_occupancy(W, L, bits, device=True, out=out)
    for _ in range(2):
        for v in out.values():
            v.zero_()
        g.replay()
        torch.cuda.synchronize()
        for k in KEYS:
            assert np.array_equal(out[k].cpu().numpy(), ref[k]), k
        assert int(out["n_percolating"][0]) == ref["n_percolating"]
