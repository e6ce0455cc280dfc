"""The wavefront solver (the default of pc_inspect): every reached site updated
once, at its first arrival.  Outputs against the oracle and against the
forced solvers (verdict, first_hit, m_stop exact; the mass within the relative
bound of the recursion's FP32 arithmetic), at the sizes where its windows,
queues and mass rings end."""
from __future__ import annotations

import os

import numpy as np
import pytest

import oracle
import paper_1401_2130_gb300 as pc

pytestmark = pytest.mark.gpu

THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    pc.build()
    pc.load()
    torch.cuda.init()


def _check(g, ref, W, what):
    """Exact verdicts and steps; mass within 1.01 (3 + 7 (first_hit - 1) +
    ceil(P / 32) + 10) 2^-24 of the FP64 oracle where it exceeds 1e-30 (the
    bound of the full recursion: each site here takes at most as many rounded
    operations), and within 1e-30 of it elsewhere."""
    for k in ("verdict", "first_hit", "m_stop"):
        assert np.array_equal(np.asarray(g[k]).astype(np.int64), np.asarray(ref[k]).astype(np.int64)), (what, k)
    if "mass" not in ref:
        return
    mg, mr = np.asarray(g["mass"], np.float64), np.asarray(ref["mass"], np.float64)
    P = pc.pc_lattice_layout(W)["P"]
    fh = np.maximum(np.asarray(ref["first_hit"]), 1)
    tol = np.where(mr > 1e-30, 1.01 * (3 + 7 * (fh - 1) + (P + 31) // 32 + 10) * 2.0 ** -24 * mr, 1e-30)
    assert np.all(np.abs(mg - mr) <= tol), what


@pytest.mark.parametrize("W,L,p,n", [
    (0, 1, 0.5, 64), (0, 700, 0.995, 40),           # one column; every level one site
    (1, 33, 0.5, 200), (3, 32, 0.4, 200), (3, 31, 0.4, 200),  # word rows full, one tube over, one short
    (5, 8, 0.3, 300), (5, 9, 0.3, 300), (5, 1, 0.3, 100),     # layers of one draw, one over
    (13, 60, 0.2, 80), (14, 60, 0.2, 80),           # one warp a configuration, one block
    (6, 400, 0.3, 60),                              # a warp's window of word rows
    (16, 130, 0.9, 40), (16, 300, 0.25, 40),        # mass rings of 128 layers
    (20, 12, 0.95, 60),                             # levels beyond the frontier queue
    (40, 70, 0.18, 24), (41, 40, 0.7, 24),          # widths of 256 and 512 threads
    (64, 140, 0.6, 6), (65, 40, 0.2, 12),           # a window of fewer rows than the lattice
    (130, 6, 0.3, 4), (140, 40, 0.17, 3),           # one word row, none, in shared memory
])
def test_against_the_oracle(W, L, p, n):
    g = pc.pc_inspect(W, L, p, 77, 5, n)
    ref = oracle.inspect(W, L, p=p, seed=77, cfg0=5, n=n, mode="markov", threads=THREADS)
    _check(g, ref, W, (W, L, p))
    assert g["n_percolating"] == int(ref["verdict"].sum())
    b = pc.pc_inspect(W, L, p, 77, 5, n, bits_only=True)
    _check(b, {k: ref[k] for k in ("verdict", "first_hit", "m_stop")}, W, "bits only")
    assert not np.any(b["mass"])
    v = pc.pc_inspect(W, L, p, 77, 5, n, verdict_first=True)
    assert np.array_equal(v["mass"], g["mass"])


@pytest.mark.parametrize("W,L,p,n", [(8, 64, 0.2, 2000), (6, 90, 0.3, 300), (20, 200, 0.19, 40), (33, 20, 0.5, 40)])
def test_masses_of_the_forced_solvers(W, L, p, n):
    """The full recursion sums the same terms with zeros in the other places;
    only the order of the final sum over the end layer differs (at most
    ceil(P / 32) + 10 additions of non-negative terms)."""
    g = pc.pc_inspect(W, L, p, 9, 0, n)
    P = pc.pc_lattice_layout(W)["P"]
    for mode in (pc.PC_MODE_RESIDENT, pc.PC_MODE_STREAM):
        try:
            f = pc.pc_inspect(W, L, p, 9, 0, n, mode=mode)
        except pc.PercolError as e:
            assert e.status == pc.PC_ERR_OOM and mode == pc.PC_MODE_RESIDENT
            continue
        for k in ("verdict", "first_hit", "m_stop"):
            assert np.array_equal(g[k], f[k]), (mode, k)
        a, b = np.asarray(g["mass"], np.float64), np.asarray(f["mass"], np.float64)
        # 2^-149 per addition where the sums are subnormal
        assert np.all(np.abs(a - b) <= 2 * ((P + 31) // 32 + 10) * (2.0 ** -24 * b + 2.0 ** -149)), mode


@pytest.mark.parametrize("W,L,p,n", [
    (24, 300, 0.18, 20),     # every word row in shared memory
    (24, 145, 0.4, 5),       # rows drawn ahead: the last step ragged
    (40, 128, 0.19, 30),     # exactly four word rows: one step
    (40, 129, 0.19, 30),     # one tube more
    (40, 700, 0.175, 12),    # three steps, a window of rows
    (64, 600, 0.17, 3),
    (46, 200, 0.9, 4),       # levels beyond the queue kept over a step
    (130, 20, 0.3, 2),       # few rows in shared memory
])
def test_rows_drawn_ahead(W, L, p, n):
    """Few configurations of large lattices: their rows are drawn ahead in
    steps, and a configuration that reaches the last drawn row goes on in the
    next launch.  Also from caller bits, and beside smaller queries."""
    import torch
    ref = oracle.inspect(W, L, p=p, seed=8, cfg0=2, n=n, mode="bfs", threads=THREADS)
    ref = {k: ref[k] for k in ("verdict", "first_hit", "m_stop")}
    g = pc.pc_inspect(W, L, p, 8, 2, n)
    _check(g, ref, W, (W, L, p))
    many = pc.pc_inspect(W, L, p, 8, 0, 200)  # drawn by the block that works on them
    for k in ("verdict", "first_hit", "m_stop", "mass"):
        assert np.array_equal(many[k][2:2 + n], g[k]), k
    bits = pc.pc_occupancy(W, L, p, 8, 2, n)
    _check(pc.pc_inspect_occupancy(W, L, bits), ref, W, "caller bits")
    outs, _ = pc.pc_batch_run([(W, L, p, 8, 2, n), (W, L // 2 + 1, p, 8, 0, 3), (4, 16, 0.2, 8, 0, 100)])
    for k in ("verdict", "first_hit", "m_stop", "mass"):
        assert np.array_equal(outs[0][k], g[k]), k
    torch.cuda.synchronize()


def _columns(W):
    return [(q, r) for r in range(-W, W + 1) for q in range(max(-W, -W - r), min(W, W - r) + 1)]


_SIDE = [(1, 1), (2, -1), (1, -2), (-1, -1), (-2, 1), (-1, 2), (1, 0), (-1, 1), (0, -1), (-1, 0), (1, -1), (0, 1)]


def _near(cols, at, L, x):
    """Contacts of site x = (tube, column)."""
    t, a = x
    q, r = cols[a]
    s = (q - r) % 3
    near = [(t - 1, a), (t + 1, a)]
    for d, (dq, dr) in enumerate(_SIDE):
        b = at.get((q + dq, r + dr))
        if b is not None:
            near.append((t + (1 if 6 <= d < 9 and s == 2 else -1 if d >= 9 and s == 0 else 0), b))
    return [y for y in near if 0 <= y[0] < L]


def _bfs_span(W, L, occ):
    """Widest range of tubes that one BFS level of each occupancy spans."""
    cols = _columns(W)
    at = {c: i for i, c in enumerate(cols)}
    A = len(cols)
    out = []
    for o in occ.reshape(len(occ), L, A).astype(bool):
        free = o.copy()
        front = [(0, a) for a in range(A) if o[0, a]]
        for x in front:
            free[x] = False
        widest = 0
        while front and max(t for t, _ in front) < L - 1:
            ts = [t for t, _ in front]
            widest = max(widest, max(ts) - min(ts) + 1)
            nxt = []
            for y in front:
                for x in _near(cols, at, L, y):
                    if free[x]:
                        free[x] = False
                        nxt.append(x)
            front = nxt
        out.append(widest)
    return np.array(out)


def _serpent(cols, at, L, start, top, keep_out, rng, length):
    """A path of up to ``length`` sites from (0, start) in the tubes below
    ``top`` whose sites touch only their neighbours along the path."""
    path = [(0, start)]
    on, blocked = {path[0]}, set()
    while len(path) < length:
        last = path[-1]
        free = [y for y in _near(cols, at, L, last)
                if 1 <= y[0] < top and y not in on and y not in blocked and y[1] not in keep_out]
        if not free:
            break
        y = free[rng.integers(len(free))]
        blocked.update(x for x in _near(cols, at, L, last) if x != y)
        path.append(y)
        on.add(y)
    return path


@pytest.mark.parametrize("W,L", [(12, 150), (30, 150), (12, 138), (30, 138)])
def test_frontiers_wider_than_windows_and_rings(W, L):
    """A straight wire up the fibre beside a long induced path in the lowest
    tubes: the levels span more tubes than the mass rings (128) and the window
    of word rows hold; in every second occupancy a branch comes back down from
    the wire's upper end."""
    import torch
    n = 6
    cols = _columns(W)
    A = len(cols)
    at = {c: i for i, c in enumerate(cols)}
    rng = np.random.default_rng(5)
    occ = np.zeros((n, L, A), np.uint8)
    wire, start = at[(-W, 0)], at[(W // 2, -W // 2)]
    keep_out = {a for a, (q, r) in enumerate(cols) if q + W <= 6}
    for k in range(n):
        path = max((_serpent(cols, at, L, start, 8, keep_out, rng, 170) for _ in range(400)), key=len)
        for x in path:
            occ[k][x] = 1
        occ[k, :, wire] = 1
        if k % 2:
            occ[k, 20:L - 4, at[(-W + 3, 0)]] = 1
            occ[k, L - 5, at[(-W + 1, 0)]] = occ[k, L - 5, at[(-W + 2, 0)]] = 1
    span = _bfs_span(W, L, occ.reshape(n, -1))
    assert span.max() > 123, span  # the rings hold a level of up to 123 tubes
    bits = torch.from_numpy(oracle.pack_bits(occ.reshape(n, -1)).view(np.int32)).cuda()
    g = pc.pc_inspect_occupancy(W, L, bits)
    ref = oracle.inspect(W, L, occ=occ.reshape(n, -1), mode="markov", threads=THREADS)
    _check(g, ref, W, ("spans", span))
    # one end-layer site carries mass: the recursion's last sum has one term,
    # and every term before it is the full recursion's to the bit
    f = pc.pc_inspect_occupancy(W, L, bits, mode=pc.PC_MODE_STREAM)
    assert np.array_equal(g["mass"], f["mass"])
    assert np.all((g["mass"] > 0) == (ref["mass"] > 2.0 ** -149))


def test_calls_on_several_streams_and_threads():
    """Scratch belongs to a call: concurrent calls on their own streams give
    the results of calls alone."""
    import threading
    import torch
    specs = [(8, 64, 0.2, 500), (20, 120, 0.19, 60), (40, 60, 0.18, 30), (4, 16, 0.3, 2000)]
    want = [pc.pc_inspect(W, L, p, 3, 0, n) for W, L, p, n in specs]
    got = [[None] * 3 for _ in specs]

    def work(i):
        W, L, p, n = specs[i]
        s = torch.cuda.Stream()
        for k in range(3):
            got[i][k] = pc.pc_inspect(W, L, p, 3, 0, n, stream=s)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(specs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for i, w in enumerate(want):
        for g in got[i]:
            for key in ("verdict", "first_hit", "m_stop", "mass"):
                assert np.array_equal(g[key], w[key]), (specs[i], key)


@pytest.mark.parametrize("W,L,p,n", [
    (52, 33, 0.9, 5), (64, 33, 0.5, 5),   # levels too large for few SMs
    (64, 32, 0.24, 9), (64, 65, 0.18, 3),  # levels for which these are the faster ones
    (90, 40, 0.25, 3),                    # a window of one row of two
    (125, 9, 0.4, 3),                     # no window row in shared memory
])
def test_the_solver_does_not_show(W, L, p, n):
    """A configuration's outputs are the same bits whatever solver a call takes:
    alone, among many, forced, in a batch beside small queries, in a server."""
    ref = pc.pc_inspect(W, L, p, 6, 0, n, mode=pc.PC_MODE_STREAM)
    many = pc.pc_inspect(W, L, p, 6, 0, 160)
    g = pc.pc_inspect(W, L, p, 6, 0, n)
    one = pc.pc_inspect(W, L, p, 6, 1, 1)
    v = pc.pc_inspect(W, L, p, 6, 0, n, verdict_first=True)
    outs, res = pc.pc_batch_run([(3, 9, 0.4, 6, 0, 50), (W, L, p, 6, 0, n)])
    assert res[1]["n_percolating"] == int(ref["verdict"].sum())
    srv = pc.Server(hbm_budget_bytes=1 << 30, max_slots=16, max_slots_per_query=4)
    try:
        t = srv.submit((W, L, p, 6, 0, n))
        served = srv.poll(t, 60.0)
        for k in ("verdict", "first_hit", "m_stop", "mass"):
            for what, o in (("many", many), ("default", g), ("verdict first", v), ("batch", outs[1]), ("server", served)):
                assert np.array_equal(np.asarray(o[k])[:n], ref[k]), (what, k)
            assert one[k][0] == ref[k][1], k
    finally:
        srv.close()
    b = pc.pc_inspect(W, L, p, 6, 0, n, bits_only=True)
    for k in ("verdict", "first_hit", "m_stop"):
        assert np.array_equal(b[k], ref[k]), k
