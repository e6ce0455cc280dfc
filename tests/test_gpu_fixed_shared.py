"""Fixed-count occupancies drawn and selected in one CTA's shared memory
against the oracle's definition, bit for bit, at the edges of the kernel's
range: each thread count's largest and next lattice, the largest lattice that
fits shared memory and the next one (which the multi-launch kernels take),
ragged words and blocks, and the extreme counts."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_1401_2130_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,L,Np,n", [
    (0, 2, 1, 5), (0, 33, 32, 700), (1, 9, 1, 300), (1, 9, 62, 300),
    (0, 1024, 200, 40), (0, 1025, 1024, 40), (0, 8192, 8191, 6), (0, 8193, 3, 6), (8, 24, 1145, 400),
    (0, 24576, 5000, 3), (0, 24577, 5000, 3), (0, 57600, 57599, 2), (0, 57601, 20000, 2), (0, 57603, 1, 2),
])
def test_selection_in_shared_memory(W, L, Np, n):
    import torch
    seed, cfg0 = 2**40 + 11, 2**31 + 5
    bits = pc.pc_occupancy_fixed(W, L, Np, seed, cfg0, n)
    torch.cuda.synchronize()
    got = bits.cpu().numpy().view(np.uint32)
    assert np.array_equal(got, oracle.pack_bits(oracle.occupancy_fixed(W, L, Np, seed, cfg0, n)))
