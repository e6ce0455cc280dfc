"""Performance cases of the percolation inspection: what users of the library
have it do, through its public entry points.

The sizes are those of the benchmark and the tests: the tiny lattice (W = 4,
L = 16), the p-sweep lattice (W = 8, L = 64), the long thin fibre of the length
scan (W = 6, p = 0.3), the largest lattice the paper inspects (W = 46,
L = 400), the large lattice (W = 64, L = 4096), the mixed batch (W in 4..32 at
several aspect ratios), the finite-size-scaling scan and the serving stream.

Outputs are verdicts, first hits and step counts (whole numbers) and the FP32
mass at the first hit; ``exact`` recomputes them with plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1401_2130_gb300 as pc
from paper_1401_2130_gb300 import fss


def _columns(W):
    return 3 * W * (W + 1) + 1


def listed():
    return [
        # the smallest call: the allocation-free entry point in a latency-critical loop
        {"name": "static_W5_L8", "kind": "static", "W": 5, "L": 8, "p": 0.25, "n": 64},
        # a first look at a lattice: one thousand configurations, host outputs
        {"name": "tiny_W4_L16", "kind": "inspect", "W": 4, "L": 16, "p": 0.15, "n": 1000, "device": False,
         "option": "full"},
        # one point of a Pi(p) curve inside the transition, device outputs
        {"name": "psweep_W8_L64", "kind": "inspect", "W": 8, "L": 64, "p": 0.185, "n": 10000, "device": True,
         "option": "full"},
        # length dependence at fixed width: a long thin fibre where nearly all configurations percolate
        {"name": "length_W6_L96", "kind": "inspect", "W": 6, "L": 96, "p": 0.3, "n": 1024, "device": True,
         "option": "full"},
        # fixed-count sampling: exactly Np metallic sites, inspected, and the lazy walk's mass
        {"name": "fixed_W8_L24", "kind": "fixed", "W": 8, "L": 24, "p": 0.22, "n": 4000, "hold": 0.3},
        # verdict first on a middling lattice near its threshold
        {"name": "first_W20_L301", "kind": "inspect", "W": 20, "L": 301, "p": 0.172, "n": 500, "device": True,
         "option": "verdict_first"},
        # the largest lattice of the paper's Fig. 3(b), 2.6 million sites
        {"name": "fibre_W46_L400", "kind": "inspect", "W": 46, "L": 400, "p": 0.165, "n": 32, "device": True,
         "option": "full"},
        # the large lattice of the benchmark, one percolating configuration
        {"name": "large_W64_L4096", "kind": "inspect", "W": 64, "L": 4096, "p": 0.17, "n": 1, "device": False,
         "option": "full"},
        # the same lattice, verdicts only
        {"name": "verdicts_W64_L4096", "kind": "inspect", "W": 64, "L": 4096, "p": 0.17, "n": 4, "device": True,
         "option": "bits_only"},
        # one submission of mixed sizes at the paper's threshold, replayed as a user with fixed buffers does
        {"name": "batch_W4_W32", "kind": "batch", "widths": "4,8,16,32", "ratios": "1,8", "p": 0.1533, "n": 400},
        # verdict counts of a finite-size-scaling scan: every size at several p
        {"name": "scan_W4_W16", "kind": "scan", "widths": "4,8,16", "ratios": "1,4,8", "ps": "0.14,0.18,0.22,0.3",
         "n": 256},
        # a burst of queries to the server
        {"name": "serve_8", "kind": "serve", "queries": 8, "stream": 5, "w_max": 32, "ratio_max": 16, "n_max": 600},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _threshold(W, L):
    """Where the transition of a W x L fibre lies, roughly (the scaling law's form)."""
    W, L = max(W, 1), max(L, 1)
    return 0.156 + 0.58 * (W / L) ** -1.22 * L ** -1.136 - 0.39 * L ** -1.136


def _sweep_cost(W, L, p, n):
    """Site visits of the plain recursion: A layers-in-window summed over its steps."""
    A = _columns(W)
    steps = 4 * L if p > _threshold(W, L) - 0.01 else min(4 * L, 40 + 8 * W)
    k = min(steps, L)
    return A * n * (k * k / 2 + (steps - k) * L + 64)


def draw(rng):
    kind = rng.choice(["inspect"] * 6 + ["static", "fixed", "batch", "scan", "serve"])

    def p_of():
        return round(rng.choice([rng.uniform(0.12, 0.19)] * 3 + [rng.uniform(0.19, 0.35), rng.uniform(0.35, 0.9)]), 4)

    if kind == "static":
        W = rng.randint(0, 8)
        return {"kind": kind, "W": W, "L": _log_int(rng, 1, 64), "p": p_of(), "n": _log_int(rng, 1, 4000)}
    if kind == "fixed":
        W = rng.randint(2, 16)
        L = _log_int(rng, max(1, W // 2), 6 * W)
        return {"kind": kind, "W": W, "L": L, "p": p_of(), "n": _log_int(rng, 16, max(17, int(6e7 / (_columns(W) * L)))),
                "hold": round(rng.uniform(0.0, 0.9), 3)}
    if kind == "batch":
        ws = sorted(rng.sample([3, 4, 6, 8, 11, 16, 23, 32], 3))
        rs = sorted(rng.sample([1, 2, 3, 4, 6, 8], 2))
        return {"kind": kind, "widths": ",".join(map(str, ws)), "ratios": ",".join(map(str, rs)),
                "p": round(rng.uniform(0.12, 0.165), 4), "n": _log_int(rng, 32, 400)}
    if kind == "scan":
        ws = sorted(rng.sample([3, 4, 5, 6, 8, 10, 12, 16], 3))
        rs = sorted(rng.sample([1, 2, 3, 4, 6, 8], 2))
        ps = sorted(round(rng.uniform(0.1, 0.5), 3) for _ in range(4))
        return {"kind": kind, "widths": ",".join(map(str, ws)), "ratios": ",".join(map(str, rs)),
                "ps": ",".join(map(str, ps)), "n": _log_int(rng, 32, 300)}
    if kind == "serve":
        return {"kind": kind, "queries": rng.randint(3, 9), "stream": rng.randint(6, 10**6),
                "w_max": rng.randint(6, 32), "ratio_max": rng.randint(2, 12), "n_max": _log_int(rng, 60, 500)}
    W = rng.choice([rng.randint(0, 16), rng.randint(4, 64), rng.randint(4, 64)])
    L = _log_int(rng, 1, 64 * max(W, 1))
    p = p_of()

    def most_of(L):  # configurations within the largest listed cases' cost
        return int(min(2.0e11 / _sweep_cost(W, L, p, 1), 3.0e9 / _one_work(W, L, p, 1)["flops"]))

    most = most_of(L)
    while most < 1:
        L = max(1, L // 2)
        most = most_of(L)
    return {"kind": "inspect", "W": W, "L": L, "p": p, "n": _log_int(rng, 1, min(10000, most)),
            "device": rng.random() < 0.6, "option": rng.choice(["full", "full", "bits_only", "verdict_first"])}


# ---------------------------------------------------------------------------
# what a user's program holds, and one pass
# ---------------------------------------------------------------------------

def _ints(text):
    return [int(x) for x in text.split(",")]


def _specs(case, seed):
    """Queries (W, L, p, seed, first configuration, configurations) of a batch, a scan or a burst."""
    kind = case["kind"]
    if kind == "batch":
        return [(W, W * r, case["p"], seed, 0, case["n"]) for W in _ints(case["widths"]) for r in _ints(case["ratios"])]
    if kind == "scan":
        return [(W, W * r, float(p), seed, 0, case["n"]) for W in _ints(case["widths"]) for r in _ints(case["ratios"])
                for p in case["ps"].split(",")]
    g = np.random.default_rng(case["stream"])
    out = []
    for k in range(case["queries"]):
        W = int(g.integers(4, case["w_max"] + 1))
        L = int(round(W * math.exp(g.uniform(0.0, math.log(case["ratio_max"])))))
        n = int(round(math.exp(g.uniform(math.log(50.0), math.log(case["n_max"])))))
        out.append((W, L, float(g.uniform(0.12, 0.19)), seed + k, 0, n))
    return out


class _Served:
    """A server that closes with the state that holds it."""

    def __init__(self):
        self.server = pc.Server(hbm_budget_bytes=16 << 30, max_slots=256, max_slots_per_query=64, max_W=64)

    def __del__(self):
        try:
            self.server.close()
        except Exception:
            pass


def prepare(case, seed):
    state = dict(case, seed=1000003 * int(seed) + 17)
    if case["kind"] == "batch":
        state["query_array"], state["outs"] = pc.batch_queries(_specs(case, state["seed"]), device=False)
    elif case["kind"] == "serve":
        state["served"] = _Served()
    return state


def _np_of(case):
    return int(case["p"] * _columns(case["W"]) * case["L"])


def run(state):
    kind, seed = state["kind"], state["seed"]
    if kind == "inspect":
        opt = state["option"]
        return pc.pc_inspect(state["W"], state["L"], state["p"], seed, 0, state["n"], device=state["device"],
                             bits_only=opt == "bits_only", verdict_first=opt == "verdict_first")
    if kind == "static":
        return pc.pc_inspect_static(state["W"], state["L"], state["p"], seed, 0, state["n"])
    if kind == "fixed":
        bits = pc.pc_occupancy_fixed(state["W"], state["L"], _np_of(state), seed, 0, state["n"])
        r = pc.pc_inspect_occupancy(state["W"], state["L"], bits, device=True)
        r["occupancy"] = bits
        r["lazy_mass"] = pc.pc_lazy_mass(r["first_hit"], r["mass"], state["hold"])
        return r
    if kind == "batch":
        outs, res = pc.pc_batch_run(_specs(state, seed), outs=state["outs"], queries=state["query_array"])
        return [dict(o) for o in outs]
    if kind == "scan":
        return np.asarray(fss.measure(_specs(state, seed)), np.int64)
    srv = state["served"].server
    tickets = [srv.submit(s) for s in _specs(state, seed)]
    out = []
    for t in tickets:
        r = None
        while r is None:
            r = srv.poll(t, 30.0)
        out.append({k: v for k, v in r.items() if k != "solver"})
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _one_work(W, L, p, n, full=True):
    # Layers that have to be looked at: all of them where the fibre percolates,
    # else those within the clusters that touch its start.
    layers = L if p > _threshold(W, L) else min(L, W + 32)
    sites = n * _columns(W) * layers
    # per site a quarter of a counter-based block (10 rounds of 2 wide
    # multiplications and 4 exclusive ors), per metallic site its 14 contacts
    return {"bytes": n * (13 if full else 9), "flops": sites * (15 + 14 * p)}


def work(case):
    kind = case["kind"]
    if kind in ("inspect", "static"):
        return _one_work(case["W"], case["L"], case["p"], case["n"])
    if kind == "fixed":
        N = _columns(case["W"]) * case["L"]
        w = _one_work(case["W"], case["L"], case["p"], case["n"])
        return {"bytes": w["bytes"] + case["n"] * (4 * ((N + 31) // 32) + 12), "flops": w["flops"] + 15 * N * case["n"]}
    parts = [_one_work(W, L, p, n) for W, L, p, _, _, n in _specs(case, 0)]
    return {"bytes": sum(x["bytes"] for x in parts), "flops": sum(x["flops"] for x in parts)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _words(W, L, seed, c0, n, dev):
    """[n, N] 32-bit words of the occupancy stream (Philox4x32-10), as int64."""
    N = _columns(W) * L
    nb = (N + 3) // 4
    m32 = 0xFFFFFFFF
    x = torch.arange(nb, dtype=torch.int64, device=dev)[None, :].expand(n, nb)
    y = torch.arange(c0, c0 + n, dtype=torch.int64, device=dev)[:, None].expand(n, nb)
    z = torch.full((1, 1), W | (L << 8), dtype=torch.int64, device=dev).expand(n, nb)
    w = torch.zeros((1, 1), dtype=torch.int64, device=dev).expand(n, nb)
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        a, b = 0xD2511F53 * x, 0xCD9E8D57 * z  # the low 64 bits, whatever the sign
        x, y, z, w = ((b >> 32) & m32) ^ y ^ k0, b & m32, ((a >> 32) & m32) ^ w ^ k1, a & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return torch.stack([x, y, z, w], -1).reshape(n, 4 * nb)[:, :N]


_SIDE = [(1, 1), (2, -1), (1, -2), (-1, -1), (-2, 1), (-1, 2), (1, 0), (-1, 1), (0, -1), (-1, 0), (1, -1), (0, 1)]


def _contacts(W, L, dev):
    """[14, A L] index of each site's contacts in planes of A + 1 columns with a
    zero layer on each side (column A is always zero)."""
    cols = [(q, r) for r in range(-W, W + 1) for q in range(max(-W, -W - r), min(W, W - r) + 1)]
    at = {c: i for i, c in enumerate(cols)}
    A = len(cols)
    t = torch.arange(1, L + 1, dtype=torch.int64, device=dev)[:, None]
    out = []
    for d, (dq, dr) in enumerate(_SIDE):
        nb = torch.tensor([at.get((q + dq, r + dr), A) for q, r in cols], dtype=torch.int64, device=dev)
        sg = torch.tensor([(q - r) % 3 for q, r in cols], dtype=torch.int64, device=dev)
        dt = (sg == 2).long() if 6 <= d < 9 else -(sg == 0).long() if d >= 9 else torch.zeros_like(sg)
        out.append(((t + dt[None, :]) * (A + 1) + nb[None, :]).reshape(-1))
    own = torch.arange(A, dtype=torch.int64, device=dev)[None, :]
    out += [((t + s) * (A + 1) + own).reshape(-1) for s in (-1, 1)]
    return torch.stack(out)


def _chain(W, L, occ):
    """The absorbing chain in FP64 for occupancies occ [n, N] (bool): verdict, first hit, mass, step count."""
    n, N = occ.shape
    A, dev = _columns(W), occ.device
    con = _contacts(W, L, dev)

    def padded(v):
        p = torch.zeros((v.shape[0], L + 2, A + 1), dtype=v.dtype, device=dev)
        p[:, 1:L + 1, :A] = v.reshape(-1, L, A)
        return p.reshape(v.shape[0], -1)

    def gather(v):
        p, s = padded(v), torch.zeros_like(v)
        for k in range(14):
            s += p[:, con[k]]
        return s

    deg = gather(occ.double())
    deg[:, N - A:] += 1.0
    inv = torch.where(occ & (deg > 0), 1.0 / deg.clamp(min=1.0), 0.0)
    start = torch.zeros_like(occ)
    start[:, :A] = occ[:, :A]
    n0 = start.sum(1)
    verdict = torch.zeros(n, dtype=torch.int64, device=dev)
    hit = torch.full((n,), -1, dtype=torch.int64, device=dev)
    mass = torch.zeros(n, dtype=torch.float64, device=dev)
    stop = torch.zeros(n, dtype=torch.int64, device=dev)
    live = torch.nonzero(n0 > 0).flatten()
    nu = (start.double() / n0.clamp(min=1)[:, None] * inv)[live]
    R, occ, inv = start[live], occ[live], inv[live]
    m = 0
    while live.numel():
        end = R[:, N - A:].any(1)  # reached the end layer: the detector is hit at the next step
        if end.any():
            i = live[end]
            verdict[i], hit[i], stop[i] = 1, m + 1, m + 1
            mass[i] = nu[end][:, N - A:].sum(1)
            keep = ~end
            live, nu, R, occ, inv = live[keep], nu[keep], R[keep], occ[keep], inv[keep]
            if not live.numel():
                break
        m += 1
        grown = R | ((gather(R.to(torch.uint8)) > 0) & occ)
        nu = gather(nu) * inv
        still = (grown == R).all(1)
        R = grown
        if still.any():
            stop[live[still]] = m
            keep = ~still
            live, nu, R, occ, inv = live[keep], nu[keep], R[keep], occ[keep], inv[keep]
    return verdict, hit, mass, stop


def _too_long(W, L, p, n):
    return _sweep_cost(W, L, p, n) > 2.5e10 or _columns(W) * L * n > 2.5e8


def _exact_inspect(W, L, p, seed, n, np_sites=None, option="full"):
    """(verdict, first_hit, mass, m_stop, occupancy) of configurations 0..n-1 as numpy arrays."""
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    N = _columns(W) * L
    chunk = max(1, int(2.5e7 / N))
    parts, bits = [], []
    for c in range(0, n, chunk):
        k = min(chunk, n - c)
        u = _words(W, L, seed & (2**64 - 1), c, k, dev)
        if np_sites is None:
            occ = u < int(p * 4294967296.0)
        else:
            key = torch.arange(N, dtype=torch.int64, device=dev)[None, :] + (u - 2**31) * 2**32
            order = key.argsort(1)[:, :np_sites]
            occ = torch.zeros((k, N), dtype=torch.bool, device=dev).scatter_(1, order, True)
            pad = torch.zeros((k, (N + 31) // 32 * 32), dtype=torch.int64, device=dev)
            pad[:, :N] = occ.long()
            word = (pad.reshape(k, -1, 32) << torch.arange(32, device=dev)).sum(-1)
            bits.append(torch.where(word >= 2**31, word - 2**32, word).to(torch.int32))
        parts.append(_chain(W, L, occ))
    v, h, m, s = (torch.cat([x[j] for x in parts]).cpu().numpy() for j in range(4))
    if option == "bits_only":
        m = np.zeros_like(m)
    return v, h, m, s, torch.cat(bits).cpu().numpy() if bits else None


def _held(mass):
    """First-passage masses shrink by the mean degree at every step; below 1e-30
    the FP32 recursion has left its normal range, so that an output without a
    larger one has no value to compare with."""
    top = mass.max(initial=0.0)
    return None if 0.0 < top < 1e-30 else mass


def exact(case, seed):
    kind, seed = case["kind"], 1000003 * int(seed) + 17
    if kind in ("inspect", "static"):
        W, L, p, n = case["W"], case["L"], case["p"], case["n"]
        if _too_long(W, L, p, n):
            return None
        v, h, m, s, _ = _exact_inspect(W, L, p, seed, n, option=case.get("option", "full"))
        out = {"verdict": v, "first_hit": h, "mass": _held(m), "m_stop": s, "n_percolating": int(v.sum())}
        if case.get("device"):
            out["n_percolating"] = np.asarray([v.sum()])
        else:
            out["Pi"] = float(v.sum()) / n
        return out
    if kind == "fixed":
        W, L, n = case["W"], case["L"], case["n"]
        if _too_long(W, L, case["p"], n):
            return None
        v, h, m, s, bits = _exact_inspect(W, L, 0.0, seed, n, np_sites=_np_of(case))
        lazy = np.where(h > 0, m * (1.0 - case["hold"]) ** h.clip(min=0), 0.0)
        return {"verdict": v, "first_hit": h, "mass": _held(m), "m_stop": s, "n_percolating": np.asarray([v.sum()]),
                "occupancy": bits, "lazy_mass": _held(lazy)}
    if kind == "scan":
        return None  # whole numbers only
    specs = _specs(case, seed)
    if sum(_sweep_cost(W, L, p, n) for W, L, p, _, _, n in specs if not _too_long(W, L, p, n)) > 5e10:
        return None
    out = []
    for W, L, p, sd, _, n in specs:
        if _too_long(W, L, p, n):
            out.append({"verdict": None, "first_hit": None, "mass": None, "m_stop": None, "n_percolating": None,
                        "Pi": None})
            continue
        v, h, m, s, _ = _exact_inspect(W, L, p, sd, n)
        out.append({"verdict": v, "first_hit": h, "mass": _held(m), "m_stop": s, "n_percolating": int(v.sum()),
                    "Pi": float(v.sum()) / n})
    return out
