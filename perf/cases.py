"""What this framework is timed on: whole iterations of the parallel multicanonical loop.

A pass is what a user's run does between two looks at its results: some iterations of the paper's
Fig. 1 loop (sweeps of every walker, merge, weight update, flatness) through the public classes,
then the results of the run: the weights, the last histogram and the checkpoint, which is the whole
updated state (walkers, weights, recursion statistics, counters).  The contexts are warmed up in
`prepare`, so that the walkers already spread over the bins as they do for most of a run.
"""
from __future__ import annotations

import json
import math
import os

import numpy as np
import torch

import paper_1312_2213_gb300 as m

SYSTEMS = {"ising": m.ISING2D, "potts": m.POTTS2D, "muma": m.ISING2D_MUMA, "polymer": m.POLYMER3D}
BETA_MUMA = 0.4407

# The paper's uneven mix: (system, L, q), 2048 walkers each.
MIX = [("ising", L, 2) for L in (16, 24, 32, 48, 64)] + [("potts", L, 10) for L in (16, 24, 32, 48)]


def _mopt(kind: str, L: int, p: int) -> int:
    """The paper's optimal iteration length, Eq. 4 (the 8-Potts fit for every q)."""
    return max(1, round((5.7 * L ** 2.51 if kind != "potts" else 24.0 * L ** 2.67) / p))


def listed():
    return [
        # The smallest run: L = 8, 64 walkers, ten iterations of the optimal length from ln W = 0,
        # with the flatness looked at after each: launches, the update and latency are what counts.
        {"name": "ising_L8_p64", "kind": "ising", "L": 8, "q": 2, "p": 64, "sweeps": _mopt("ising", 8, 64),
         "iterations": 10, "record": 0, "observables": 0, "warm": 0, "warm_sweeps": 0},
        # A ragged walker count, magnetisation sums recorded: a small production run.
        {"name": "ising_L24_p1000_obs", "kind": "ising", "L": 24, "q": 2, "p": 1000, "sweeps": 97,
         "iterations": 5, "record": 0, "observables": 1, "warm": 12, "warm_sweeps": 40},
        # The headline configuration: L = 32, 8192 walkers, long iterations.
        {"name": "ising_L32_p8192", "kind": "ising", "L": 32, "q": 2, "p": 8192, "sweeps": 2000,
         "iterations": 1, "record": 0, "observables": 0, "warm": 20, "warm_sweeps": 40},
        # Its multimagnetic half (weights in M at fixed beta).
        {"name": "muma_L32_p8192", "kind": "muma", "L": 32, "q": 2, "p": 8192, "sweeps": 2000,
         "iterations": 1, "record": 0, "observables": 0, "warm": 20, "warm_sweeps": 40},
        # The first-order Potts configuration.
        {"name": "potts8_L32_p8192", "kind": "potts", "L": 32, "q": 8, "p": 8192, "sweeps": 2000,
         "iterations": 1, "record": 0, "observables": 0, "warm": 30, "warm_sweeps": 50},
        # The largest lattice: q = 10, L = 64 (threshold table larger than shared memory).
        {"name": "potts10_L64_p8192", "kind": "potts", "L": 64, "q": 10, "p": 8192, "sweeps": 400,
         "iterations": 1, "record": 0, "observables": 0, "warm": 10, "warm_sweeps": 40},
        # The uneven mix as one graph of short iterations: updates and launches weigh in.
        {"name": "mix_short", "kind": "mix", "p": 2048, "sweeps": 10, "iterations": 20, "warm": 10, "scale": 1.0},
        # The mix with every system at its own optimal iteration length.
        {"name": "mix_mopt", "kind": "mix", "p": 2048, "sweeps": 0, "iterations": 3, "warm": 10, "scale": 1.0},
        # The short chain and the longest one of the polymer configuration (pilot windows).
        {"name": "polymer_N13_p4096", "kind": "polymer", "N": 13, "p": 4096, "model": 0, "moves": 0, "sweeps": 400,
         "iterations": 2, "warm": 6, "warm_sweeps": 40},
        {"name": "polymer_N128_p4096", "kind": "polymer", "N": 128, "p": 4096, "model": 0, "moves": 0, "sweeps": 100,
         "iterations": 2, "warm": 4, "warm_sweeps": 20},
        # The paper's own polymer: its potentials, shifts mixed with spherical rotations.
        {"name": "polymer_N40_paper", "kind": "polymer", "N": 40, "p": 4096, "model": 1, "moves": 1, "sweeps": 60,
         "iterations": 2, "warm": 4, "warm_sweeps": 20},
        # Closing an iteration of a sharded run with the exchanged histogram (no sweeps), then
        # reweighting it (Eq. 2): the update path at the largest bin count.
        {"name": "update_potts10_L64", "kind": "update", "L": 64, "q": 10, "beta": 1.4},
    ]


def draw(rng):
    kind = rng.choice(["ising", "ising", "muma", "potts", "potts", "polymer", "polymer", "mix", "update"])
    if kind == "mix":
        return {"kind": "mix", "p": int(round(2 ** rng.uniform(8, 11))), "sweeps": rng.choice([0, 3, 10, 25]),
                "iterations": rng.randint(1, 5), "warm": 6, "scale": rng.choice([0.25, 0.5, 1.0])}
    if kind == "update":
        return {"kind": "update", "L": rng.choice([8, 16, 24, 32, 48, 64]), "q": rng.randint(3, 16),
                "beta": rng.uniform(0.8, 1.6)}
    if kind == "polymer":
        N = int(round(2 ** rng.uniform(2, 7)))
        p = int(round(2 ** rng.uniform(6, 12)))
        model = rng.choice([0, 0, 1])
        # at most about the attempts of the listed N = 128 chain, and its serial length
        sweeps = max(2, min(int(10 ** rng.uniform(6.0, 7.7) / (p * N)), 12800 // N))
        return {"kind": "polymer", "N": N, "p": p, "model": model, "moves": rng.choice([0, 0, model]),
                "sweeps": sweeps, "iterations": rng.randint(1, 2), "warm": 3, "warm_sweeps": 10}
    L = rng.choice([8, 16, 24, 32, 48, 64])
    p = int(round(2 ** rng.uniform(6, 13)))
    # attempts from short iterations to those of the listed cases, and at most their serial length
    sweeps = max(1, min(int(10 ** rng.uniform(6.0, 10.1) / (p * L * L)), 1500 * 1024 // (L * L)))
    return {"kind": kind, "L": L, "q": rng.randint(3, 12) if kind == "potts" else 2, "p": p, "sweeps": sweeps,
            "iterations": 1, "record": rng.choice([0, 0, 0, 1]),
            "observables": rng.choice([0, 1]) if kind == "ising" else 0, "warm": 6, "warm_sweeps": 20}


# ---- inputs ------------------------------------------------------------------------------------
def _seed(seed: int, i: int = 0) -> int:
    return (int(seed) * 1000003 + 17 * i + 1) & 0x7FFFFFFFFFFF


def _window(N: int, model: int):
    """The packaged pilot window of this length, else one interpolated per bead between them."""
    with open(os.path.join(os.path.dirname(os.path.abspath(m.__file__)), "polymer_windows.json")) as f:
        d = json.load(f)
    w = d["windows"] if model == 0 else d["paper_model"]["windows"]
    ns = sorted(int(k) for k in w)
    if str(N) in w:
        return (w[str(N)]["e_lo"], w[str(N)]["e_hi"])
    lo, hi = (float(np.interp(N, ns, [w[str(k)][e] / k for k in ns])) * N for e in ("e_lo", "e_hi"))
    return (math.floor(10 * lo) / 10, math.ceil(10 * hi) / 10)


def _lattice(kind, L, q, p, seed, record=0, observables=0):
    c = m.Muca(SYSTEMS[kind], L, q, p, seed, beta=BETA_MUMA if kind == "muma" else None, record=record)
    if observables:
        c.set_param("observables", 1)
    return c


def _mix_sweeps(case):
    """Sweeps of every mix system: one number for all, or each system's own optimal length."""
    if case["sweeps"]:
        return [case["sweeps"]] * len(MIX)
    return [max(1, round(case["scale"] * _mopt(k, L, 2048))) for k, L, _ in MIX]


def _histogram(B: int, reach: np.ndarray, seed: int) -> np.ndarray:
    """Counts as a nearly converged run merges them: broad, noisy, empty at the upper end."""
    r = np.random.default_rng(seed)
    x = np.linspace(-1.0, 1.0, B)
    mean = 4.0e5 * np.exp(-0.5 * (x / 0.6) ** 2)
    h = r.poisson(mean * r.gamma(30.0, 1.0 / 30.0, B)).astype(np.uint64)
    h[B - B // 64:] = 0
    h[~reach] = 0
    return h


def _potts_reach(L: int) -> np.ndarray:
    """Bins of a q >= 3 Potts lattice that some state has (bin = number of unequal bonds)."""
    reach = np.ones(2 * L * L + 1, dtype=bool)
    reach[[1, 2, 3, 5]] = False
    return reach


def prepare(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    if kind == "update":
        c = m.Muca(m.POTTS2D, case["L"], case["q"], 32, _seed(seed))
        reach = _potts_reach(case["L"])
        # an earlier iteration is already in the accumulated statistics
        h = [torch.from_numpy(_histogram(c.B, reach, _seed(seed, i)).astype(np.int64)).cuda() for i in range(2)]
        c.update_with(h[0])
        c.synchronize()
        return {"case": case, "c": c, "h": h[1]}
    if kind == "mix":
        cs = [_lattice(k, L, q, case["p"], _seed(seed, i)) for i, (k, L, q) in enumerate(MIX)]
        b = m.Batch(cs)
        b.set_sweeps(_mix_sweeps(case))
        b.run(case["warm"], 1, use_graph=False)
        b.run(case["iterations"], 1, use_graph=True)  # the program's graph is captured here
        for c in cs:
            c.synchronize()
        return {"case": case, "cs": cs, "b": b}
    if kind == "polymer":
        c = m.Muca(m.POLYMER3D, case["N"], 0, case["p"], _seed(seed), window=_window(case["N"], case["model"]))
        if case["model"]:
            c.set_param("model", case["model"])
        if case["moves"]:
            c.set_param("moves", case["moves"])
    else:
        c = _lattice(kind, case["L"], case["q"], case["p"], _seed(seed), case["record"], case["observables"])
    for _ in range(case["warm"]):
        c.iterate(case["warm_sweeps"])
        c.merge_and_update()
    c.synchronize()
    return {"case": case, "c": c}


# ---- one pass ----------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "update":
        c = state["c"]
        flat = c.update_with(state["h"], want_flat=True)
        avg, lnP = c.reweight(case["beta"])
        return {"flat": int(flat), "lnW": c.lnW(), "stats": c.flatness(), "averages": avg, "lnP": lnP}
    if kind == "mix":
        state["b"].run(case["iterations"], 1, use_graph=True)
        return {"lnW": [c.lnW() for c in state["cs"]], "H": [c.histogram() for c in state["cs"]],
                "state": [c.get_state() for c in state["cs"]]}
    c = state["c"]
    flat = []
    for _ in range(case["iterations"]):
        c.iterate(case["sweeps"])
        flat.append(int(c.merge_and_update(want_flat=True)))
    out = {"flat": flat, "lnW": c.lnW(), "H": c.histogram(), "state": c.get_state()}
    if case.get("observables"):
        out["sums"] = c.observables(0.44)[1]
    return out


# ---- what a pass cannot do without -------------------------------------------------------------
def _lattice_work(kind, L, p, attempts):
    bits = 4 if kind == "potts" else 1
    B = 2 * L * L + 1 if kind == "potts" else L * L + 1
    # lattice and bin of every walker read and written once; weights, statistics, histogram
    return 2 * (p * L * L * bits // 8 + 4 * p) + 48 * B, 30 * attempts


def work(case):
    """Bytes of the state read and written once; operations: about 30 a lattice attempt (random
    word, neighbour count, threshold, compare, update, visit) and, for the polymer, 21 a pair
    (separation 8, energy 12, sum 1), with every pair of the moved bead before and after."""
    kind = case["kind"]
    if kind == "update":
        B = 2 * case["L"] ** 2 + 1
        return {"bytes": B * (8 + 16 + 8 + 4 * 9 + 8), "flops": B * (60 + 9 * 40 + 80)}
    if kind == "mix":
        by = fl = 0
        for (k, L, _), s in zip(MIX, _mix_sweeps(case)):
            b, f = _lattice_work(k, L, case["p"], case["p"] * L * L * s * case["iterations"])
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    if kind == "polymer":
        n = case["p"] * case["N"] * case["sweeps"] * case["iterations"]
        lo, hi = _window(case["N"], case["model"])
        return {"bytes": 2 * case["p"] * (24 * case["N"] + 12) + 48 * int(10 * (hi - lo) + 1),
                "flops": n * 2 * (case["N"] - 1) * 21}
    b, f = _lattice_work(kind, case["L"], case["p"],
                         case["p"] * case["L"] ** 2 * case["sweeps"] * case["iterations"])
    return {"bytes": b, "flops": f}


# ---- the same in plain 64-bit numpy ------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on arrays of counters."""
    M, lo32 = (np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)), np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = M[0] * c[0], M[1] * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & lo32, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & lo32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack(c, axis=-1)


def _accumulate(h, rl, G, lnR):
    """One accumulated-statistics step over the ordered reachable bins; returns ln W."""
    h0, h1 = h[rl[:-1]].astype(float), h[rl[1:]].astype(float)
    ok = (h0 > 0) & (h1 > 0)
    g = h0[ok] * h1[ok] / (h0[ok] + h1[ok])
    G[ok] += g
    lnR[ok] += g / G[ok] * (np.log(h0[ok]) - np.log(h1[ok]))
    lnW = np.full(h.size, -np.inf)
    lnW[rl] = np.concatenate([[0.0], np.cumsum(lnR)])
    return lnW


def _exact_lattice(case, seed):
    L, p, N = case["L"], case["p"], case["L"] ** 2
    muma = case["kind"] == "muma"
    seed = _seed(seed)
    w = np.arange(p)
    u = _philox(np.arange(N // 4)[:, None], 0, w[None, :], 0, seed)  # word i % 4 of group i // 4
    s = np.where(u.transpose(0, 2, 1).reshape(N, p) >> np.uint64(31), -1, 1).astype(np.int64)
    lat = s.reshape(L, L, p)
    if muma:
        b = (s.sum(0) + N) // 2
    else:
        b = (-(lat * (np.roll(lat, -1, 0) + np.roll(lat, -1, 1))).sum((0, 1)) + 2 * N) // 4
    reach = np.ones(N + 1, dtype=bool)
    if not muma:
        reach[[1, N - 1]] = False
    rl = np.flatnonzero(reach)
    G, lnR, lnW = np.zeros(rl.size - 1), np.zeros(rl.size - 1), np.where(reach, 0.0, -np.inf)
    flat, g = [], 0
    plan = [case["warm_sweeps"]] * case["warm"] + [case["sweeps"]] * case["iterations"]
    nb = [(i // L * L + (i % L + 1) % L, i // L * L + (i % L - 1) % L, (i + L) % N, (i - L) % N) for i in range(N)]
    for it, sweeps in enumerate(plan):
        h = np.zeros(N + 1, dtype=np.uint64)
        for _ in range(sweeps):
            u = _philox(np.arange(N // 4)[:, None], g, w[None, :], 1, seed).transpose(0, 2, 1).reshape(N, p)
            visits = np.zeros((N, p), dtype=np.int64)
            for i in range(N):
                r, l, d, t = nb[i]
                dE = 2 * s[i] * (s[r] + s[l] + s[d] + s[t])
                b2 = np.clip(b - s[i] if muma else b + dE // 4, 0, N)
                x = np.where(reach[b2], np.where(reach[b2], lnW[b2], 0.0) - lnW[b], -np.inf)
                if muma:
                    x = x - BETA_MUMA * dE
                acc = (x >= 0) | (u[i] < np.floor(4294967296.0 * np.exp(np.minimum(x, 0.0))))
                s[i] = np.where(acc, -s[i], s[i])
                b = np.where(acc, b2, b)
                visits[i] = b
            h += np.bincount((visits if case["record"] == 0 else visits[-1]).ravel(), minlength=N + 1).astype(np.uint64)
            g += 1
        lnW = _accumulate(h, rl, G, lnR)
        if it >= case["warm"]:
            hr = h[rl]
            flat.append(int(hr.min() > 0 and hr.min() / hr.mean() >= 0.5))
    return {"flat": flat, "lnW": lnW, "H": h, "state": None}


def exact(case, seed):
    if case["kind"] == "update":
        N, beta = case["L"] ** 2, case["beta"]
        reach = _potts_reach(case["L"])
        rl = np.flatnonzero(reach)
        G, lnR = np.zeros(rl.size - 1), np.zeros(rl.size - 1)
        h = [_histogram(reach.size, reach, _seed(seed, i)) for i in range(2)]
        sampled = _accumulate(h[0], rl, G, lnR)
        lnW = _accumulate(h[1], rl, G, lnR)
        hr = h[1][rl].astype(float)
        E = np.arange(reach.size) - 2.0 * N
        seen = h[1] > 0
        x = np.full(reach.size, -np.inf)
        x[seen] = np.log(h[1][seen].astype(float)) - sampled[seen] - beta * E[seen]
        top = x.max()
        lse = top + math.log(np.exp(x - top).sum())
        P = np.exp(x - lse)
        e1, e2 = (P * E).sum(), (P * E * E).sum()
        # ln Z normalised by the ground state's degeneracy q (bin 0, E = -2 N)
        lnZ = lse + math.log(case["q"]) - (x[0] - beta * 2.0 * N) if seen[0] else float("nan")
        return {"flat": int(hr.min() > 0 and hr.min() / hr.mean() >= 0.5), "lnW": lnW,
                "stats": np.array([hr.min(), hr.mean(), hr.max()]),
                "averages": np.array([e1, e2, beta * beta * (e2 - e1 * e1) / N, lnZ]), "lnP": x - lse}
    if case["kind"] in ("ising", "muma") and not case["observables"]:
        sites = case["L"] ** 2 * (case["warm"] * case["warm_sweeps"] + case["iterations"] * case["sweeps"])
        if sites <= 60000 and sites * case["p"] <= 2e7:
            return _exact_lattice(case, seed)
    return None
