"""The work users of this library have it do, as timed cases.

Every case goes through the public binding with the library's default launch
shape, as the drivers of the package do (iterate, production, tempering,
condensation, scaling, seeding).  Sizes are those of the workloads, the
studies and the README of this repository.  Random numbers are counter-based,
so a case's integers depend on its seed alone.
"""
import math

import numpy as np
import torch

from paper_1401_4076_gb300 import mucal as m
from paper_1401_4076_gb300 import workloads

OPS = {2: 84, 3: 88}   # integer operations of one attempted move (Philox block,
                       # index maps, list reads, occupancy tests, compare, record)


def listed():
    return [
        # the README's quick start and the smoke check: one short iteration of a
        # tiny gas with its weight update; launches and round trips count
        {"name": "iterate-2d16", "kind": "iterate", "d": 2, "L": 16, "N": 32, "walkers": 64, "sweeps": 20},
        # the 2D workload of the learned-seeding and flatness studies, one of the
        # hundreds of iterations to a flat histogram
        {"name": "iterate-2d64", "kind": "iterate", "d": 2, "L": 64, "N": 410, "walkers": 4096, "sweeps": 50},
        # the 3D workload: lists of all walkers larger than L2
        {"name": "iterate-3d32", "kind": "iterate", "d": 3, "L": 32, "N": 3277, "walkers": 8192, "sweeps": 20},
        # the larger seeding target: more than 65536 sites, 32-bit site lists
        {"name": "iterate-3d48", "kind": "iterate", "d": 3, "L": 48, "N": 11059, "walkers": 2048, "sweeps": 4},
        # the walker-count study (tunnelling events decide convergence), odd lattice
        {"name": "tunnel-2d74", "kind": "tunnel", "d": 2, "L": 74, "N": 100, "walkers": 1024, "sweeps": 137},
        # the benchmark's 27 uneven systems in one launch, weights of all updated
        {"name": "batch-27", "kind": "batch", "walkers": 16384, "sweeps": 10},
        # one round of the tempering run that finds an energy window: canonical
        # update of an 8-temperature ladder, exchanges, histograms
        {"name": "temper-3d21", "kind": "temper", "d": 3, "L": 21, "N": 100, "walkers": 256, "sweeps": 5,
         "temps": 8, "T": 0.5},
        # one production round of the condensation study: five lattice sizes of
        # one particle number, histograms and the largest droplet of every walker
        {"name": "condense-2d", "kind": "condense", "N": 100, "Lmin": 61, "Lmax": 97, "systems": 5,
         "walkers": 1024, "sweeps": 50},
        # the droplet measurement alone on the 3D workload's walkers
        {"name": "droplets-3d32", "kind": "droplets", "d": 3, "L": 32, "N": 3277, "walkers": 8192},
        # a program's start: device state, initial placement, a first short iteration
        {"name": "start-3d32", "kind": "start", "d": 3, "L": 32, "N": 3277, "walkers": 8192, "sweeps": 1},
        # the seeding network proposing weights for every energy of 3D L=48
        {"name": "net-forward", "kind": "forward", "d": 3, "L": 48, "N": 11059},
        # the seeding network's training on the converged small systems
        {"name": "net-train", "kind": "train", "rows": 7001, "steps": 50},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _gas(rng, walkers_hi, attempts_hi):
    """One lattice gas of the declared ranges: 2D L 12..256, 3D L 6..48, density
    1.5 to 13 per cent, 16 walkers and more, at most 60000 attempts a walker and
    attempts_hi in all."""
    d = rng.choice((2, 3))
    L = _log(rng, 12, 256) if d == 2 else _log(rng, 6, 48)
    N = max(4, int(round(rng.uniform(0.015, 0.13) * L ** d)))
    walkers = min(_log(rng, 16, walkers_hi), int(1.2e9 / L ** d), max(1, attempts_hi // (2 * N)))
    sweeps = max(1, min(_log(rng, 2, 500), 60000 // N, attempts_hi // (N * walkers)))
    return {"d": d, "L": L, "N": N, "walkers": walkers, "sweeps": sweeps}


def draw(rng):
    kind = rng.choice(("iterate",) * 5 + ("tunnel", "batch", "temper", "condense", "droplets", "start",
                                          "forward", "gradients", "train"))
    if kind == "iterate":
        return dict(_gas(rng, 16384, 200_000_000), kind=kind)
    if kind == "tunnel":
        return {"kind": kind, "d": 2, "L": rng.randint(40, 90), "N": rng.randint(60, 200),
                "walkers": _log(rng, 64, 4096), "sweeps": rng.randint(5, 100)}
    if kind == "batch":
        return {"kind": kind, "walkers": _log(rng, 2000, 16000), "sweeps": rng.randint(2, 9)}
    if kind == "temper":
        d = rng.choice((2, 3))
        return {"kind": kind, "d": d, "L": rng.randint(40, 100) if d == 2 else rng.randint(14, 30),
                "N": rng.randint(60, 220), "walkers": _log(rng, 64, 1024), "sweeps": rng.randint(2, 12),
                "temps": rng.randint(4, 10), "T": 0.375 if d == 2 else 0.5}
    if kind == "condense":
        lo = rng.randint(50, 90)
        return {"kind": kind, "N": rng.randint(80, 200), "Lmin": lo, "Lmax": lo + rng.randint(8, 50),
                "systems": rng.randint(2, 6), "walkers": _log(rng, 128, 1024), "sweeps": rng.randint(10, 60)}
    if kind in ("droplets", "start"):
        c = dict(_gas(rng, 8192, 40_000_000), kind=kind)
        c["walkers"] = max(1, min(c["walkers"], int(2.6e8 / c["L"] ** c["d"])))
        if kind == "droplets":
            del c["sweeps"]
        else:
            c["sweeps"] = 1
        return c
    if kind == "forward":
        d = rng.choice((2, 3))
        L = _log(rng, 16, 256) if d == 2 else _log(rng, 8, 48)
        return {"kind": kind, "d": d, "L": L, "N": max(4, int(round(rng.uniform(0.04, 0.1) * L ** d)))}
    if kind == "gradients":
        return {"kind": kind, "rows": _log(rng, 100, 20000)}
    return {"kind": kind, "rows": _log(rng, 200, 7000), "steps": rng.randint(5, 49)}


# ---------------------------------------------------------------- preparation

def _seed_base(seed):
    return 1_000_003 * int(seed) + 17


def _spread(case):
    n = case["systems"]
    Ls = [case["Lmin"] + round(i * (case["Lmax"] - case["Lmin"]) / max(1, n - 1)) for i in range(n)]
    return sorted(set(Ls))


def _systems(case, seed=0):
    """System descriptors of a simulation case over the whole energy range."""
    base, w = _seed_base(seed), case["walkers"]
    if case["kind"] == "batch":
        return list(workloads.batched_uneven(w, base).systems)
    if case["kind"] == "temper":
        return [(case["d"], case["L"], case["N"], w, 0, 0, base + k * w) for k in range(case["temps"])]
    if case["kind"] == "condense":
        return [(2, L, case["N"], w, 0, 0, base + i * w) for i, L in enumerate(_spread(case))]
    return [(case["d"], case["L"], case["N"], w, 0, 0, base)]


WARM = 3   # iterations of the weight recursion behind a timed one


def _net_data(case, seed):
    """Parameters (fan-in uniform, the flat fp32 vector), rows and targets."""
    rng = np.random.default_rng(_seed_base(seed))
    parts = []
    for n, fan in ((512, 4), (128, 4), (16384, 128), (128, 128), (128, 128), (1, 128)):
        lim = 1.0 / math.sqrt(fan)
        parts.append(rng.uniform(-lim, lim, size=n))
    params = np.concatenate(parts).astype(np.float32)
    if case["kind"] == "forward":
        d, L, N = case["d"], case["L"], case["N"]
        V = L ** d
        e = np.arange(-d * N, 1) / V
        X = np.empty((len(e), 4), dtype=np.float32)
        X[:, 0], X[:, 1] = 2.0 * (d - 2.5), 16.0 / L
        X[:, 2], X[:, 3] = 10.0 * N / V - 0.5, 2.0 * e * V / (d * N) + 1.0
        return params, X, None
    # rows like the converged small systems': a few sizes and densities, all energies
    n = case["rows"]
    X = np.empty((n, 4), dtype=np.float32)
    X[:, 0] = rng.choice((-1.0, 1.0), n)
    X[:, 1] = 16.0 / rng.choice((6, 8, 10, 12, 14, 16, 20, 24, 28, 32, 40), n)
    X[:, 2] = 10.0 * rng.choice((0.05, 0.07, 0.09, 0.1, 0.11, 0.13), n) - 0.5
    X[:, 3] = rng.uniform(-1.0, 1.0, n)
    t = (0.75 + 0.2 * X[:, 3] - 0.1 * X[:, 3] ** 2 + 0.03 * X[:, 0] * X[:, 1]
         + 0.01 * rng.normal(size=n)).astype(np.float32)
    return params, X, t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients", "train"):
        params, X, t = _net_data(case, seed)
        return {"case": case, "net": m.Mlp(params), "X": X, "t": t}
    st = {"case": case, "systems": _systems(case, seed), "it": 0}
    if kind == "start":
        return st
    mc = st["mc"] = m.Mucal(st["systems"])
    n = len(st["systems"])
    if kind == "temper":
        b = np.geomspace(1.0 / (0.85 * case["T"]), 1.0 / (2.0 * case["T"]), case["temps"])
        st["betas"] = b
        grid = np.arange(-case["d"] * case["N"], 1, dtype=np.float64)
        for k in range(n):
            mc.set_weights(k, -b[k] * grid)
    elif kind == "droplets":
        # bonds favoured: droplets form
        mc.set_weights(0, -1.2 * np.arange(case["d"] * case["N"] + 1, dtype=np.float64))
    if kind == "tunnel":
        mc.set_tunnel_window(0, -case["N"] // 2, 0)
    for _ in range(WARM):
        _iterate(st, update=kind not in ("temper", "droplets"), sweeps=case.get("sweeps", 5))
    return st


def _iterate(st, update=True, sweeps=None):
    mc = st["mc"]
    mc.run_iteration(sweeps, st["it"])
    st["it"] += 1
    return [mc.update_weights(k) for k in range(len(st["systems"]))] if update else None


# ------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return state["net"].forward(state["X"])
    if kind == "gradients":
        loss, g = state["net"].gradients(state["X"], state["t"])
        return {"loss": loss, "grad": g}
    if kind == "train":
        loss = state["net"].train(state["X"], state["t"], case["steps"], 2e-3)
        return {"loss": loss, "params": state["net"].params()}
    if kind == "start":
        with m.Mucal(state["systems"]) as mc:
            mc.run_iteration(case["sweeps"], 0)
            return mc.histogram(0)
    mc = state["mc"]
    n = len(state["systems"])
    if kind == "iterate":
        (lnW, flat), = _iterate(state, sweeps=case["sweeps"])
        return {"H": mc.histogram(0), "lnW": lnW, "flat": flat}
    if kind == "tunnel":
        (lnW, flat), = _iterate(state, sweeps=case["sweeps"])
        total, per, ends = mc.tunnel_counts(0)
        return {"H": mc.histogram(0), "lnW": lnW, "events": total, "per": per.astype(np.int64), "ends": ends}
    if kind == "batch":
        up = _iterate(state, sweeps=case["sweeps"])
        return {"H": [mc.histogram(k) for k in range(n)], "lnW": [w for w, _ in up],
                "flat": np.array([f for _, f in up])}
    if kind == "temper":
        _iterate(state, update=False, sweeps=case["sweeps"])
        acc = mc.replica_exchange(state["betas"], state["it"], state["it"] % 2)
        return {"accepted": acc, "H": [mc.histogram(k) for k in range(n)]}
    if kind == "condense":
        _iterate(state, update=False, sweeps=case["sweeps"])
        H = [mc.histogram(k) for k in range(n)]
        mc.measure_droplets()
        return {"H": H, "droplets": [mc.droplet_stats(k) for k in range(n)]}
    mc.reset_droplet_stats()
    mc.measure_droplets()
    return {"stats": mc.droplet_stats(0), "largest": mc.largest_droplets(0)}


# -------------------------------------------------------------- what it takes

def work(case):
    kind = case["kind"]
    if kind == "forward":
        B = case["d"] * case["N"] + 1
        return {"bytes": B * 20 + 17281 * 4, "flops": B * 2 * (4 * 128 + 128 * 128 + 128)}
    if kind in ("gradients", "train"):
        B, steps = case["rows"], case.get("steps", 1)
        # parameters and Adam state in and out each step, rows read each step
        return {"bytes": steps * (B * 20 + 17281 * 4 * (6 if kind == "train" else 2)),
                "flops": steps * B * 6 * (4 * 128 + 128 * 128 + 128)}
    b = f = 0
    for d, L, N, W, _, _, _ in _systems(case):
        V, bins = L ** d, d * N + 1
        ib = 2 if V <= 65536 else 4
        if kind == "droplets":
            b += W * (N * ib + V // 8 + 8) + 3 * 8 * bins
            f += W * N * 3 * d
            continue
        A = case["sweeps"] * N
        # list entries and occupation words an iteration can touch, in and out
        # (a start writes all of them), the thresholds in, the histogram out
        seen = V if kind == "start" else min(V, 2 * A)
        b += W * (2 * seen * ib + 2 * min(V // 8, 8 * A) + 8) + bins * ((4 * d + 1) * 4 + 8)
        f += W * A * OPS[d]
        if kind == "temper":
            b += W * (V * ib + V // 8)   # half the replicas in a pair, swapped or not
        if kind == "condense":
            b += W * (N * ib + V // 8 + 8) + 3 * 8 * bins
            f += W * N * 3 * d
    return {"bytes": b, "flops": f}


# ------------------------------------------------- 64-bit values of the outputs

def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients", "train"):
        if kind != "forward" and case["rows"] * case.get("steps", 1) > 500_000:
            return None
        return _net_exact(case, seed)
    if kind == "iterate":
        # one numpy step per attempt, all walkers at once
        attempts = (WARM + 1) * case["sweeps"] * case["N"]
        if attempts * (1.5e-4 + 8e-7 * case["walkers"]) < 15 and case["walkers"] * case["L"] ** case["d"] < 3e7:
            return _chain_exact(case, seed)
    return None


def _net_exact(case, seed):
    params, X, t = _net_data(case, seed)
    w = torch.from_numpy(params).double()
    X = torch.from_numpy(X).double()
    rounded = lambda v: v.float().bfloat16().double()  # noqa: E731  the weights the network computes with

    def net(p):
        W1, b1, W2, b2, W3, b3 = torch.split(p, [512, 128, 16384, 128, 128, 1])
        g = torch.nn.functional.gelu
        h = g(X @ W1.view(128, 4).T + b1)
        return g(h @ W2.view(128, 128).T + b2) @ W3 + b3
    if case["kind"] == "forward":
        return net(rounded(w)).numpy()
    t = torch.from_numpy(t).double()

    def gradient(p):
        p = rounded(p).requires_grad_(True)
        loss = ((net(p) - t) ** 2).mean()
        loss.backward()
        return loss.item(), p.grad
    if case["kind"] == "gradients":
        loss, g = gradient(w)
        return {"loss": loss, "grad": g.numpy()}
    m1, m2 = torch.zeros_like(w), torch.zeros_like(w)
    for s in range(1, case["steps"] + 1):
        loss, g = gradient(w)
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        w = w - 2e-3 * (m1 / (1 - 0.9 ** s)) / ((m2 / (1 - 0.999 ** s)).sqrt() + 1e-8)
    return {"loss": loss, "params": w.numpy()}


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on arrays of 32-bit words held in 64 bits."""
    low = np.uint64(0xFFFFFFFF)
    c0, c1, c2, c3, k0, k1 = (np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3, k0, k1))
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = (p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & low, (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & low
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & low, (k1 + np.uint64(0xBB67AE85)) & low
    return c0, c1, c2, c3


def _chain_exact(case, seed):
    d, L, N, W = case["d"], case["L"], case["N"], case["walkers"]
    V, nb = L ** d, d * N + 1
    key = np.uint64(_seed_base(seed)) + np.arange(W, dtype=np.uint64)
    k0, k1 = key & np.uint64(0xFFFFFFFF), key >> np.uint64(32)
    up32 = np.uint64(32)
    s = np.arange(V)
    nbr = np.empty((V, 2 * d), dtype=np.int64)
    for k in range(d):
        x = s // L ** k % L
        nbr[:, 2 * k] = s + np.where(x == 0, L - 1, -1) * L ** k
        nbr[:, 2 * k + 1] = s + np.where(x == L - 1, 1 - L, 1) * L ** k
    all_w = np.arange(W)
    S = np.tile(s, (W, 1))
    for j in range(N):                                   # partial Fisher-Yates placement
        r = _philox(j // 4, 0, 0, 1, k0, k1)[j % 4]
        idx = j + (r * np.uint64(V - j) >> up32).astype(np.int64)
        S[all_w, j], S[all_w, idx] = S[all_w, idx], S[all_w, j].copy()
    occ = np.zeros((W, V), dtype=np.int64)
    occ[all_w[:, None], S[:, :N]] = 1
    E = -(occ * occ[:, nbr[:, 1::2]].sum(axis=2)).sum(axis=1)
    lnW, visited, pacc = np.zeros(nb), np.zeros(nb, dtype=bool), np.zeros(nb)
    for it in range(WARM + 1):
        T = np.zeros((nb, 4 * d + 1), dtype=np.int64)    # acceptance min(1, W'/W) in units of 2^-32
        for j in range(4 * d + 1):
            b = np.arange(max(0, 2 * d - j), min(nb, nb + 2 * d - j))
            diff = lnW[b + j - 2 * d] - lnW[b]
            T[b, j] = np.where(diff >= 0, 2 ** 32,
                               np.minimum(np.floor(2.0 ** 32 * np.exp(np.minimum(diff, 0))), 2 ** 32 - 2))
        H = np.zeros(nb, dtype=np.int64)
        for step in range(case["sweeps"] * N):
            r = _philox(step, 0, it, 0, k0, k1)
            k = (r[0] * np.uint64(N) >> up32).astype(np.int64)
            h = N + (r[1] * np.uint64(V - N) >> up32).astype(np.int64)
            a, b = S[all_w, k], S[all_w, h]
            near = occ[all_w[:, None], nbr[b]].sum(axis=1) - (nbr[b] == a[:, None]).sum(axis=1)
            dE = occ[all_w[:, None], nbr[a]].sum(axis=1) - near
            ok = r[2].astype(np.int64) < T[E + nb - 1, dE + 2 * d]
            w = all_w[ok]
            S[w, k[ok]], S[w, h[ok]] = b[ok], a[ok]
            occ[w, a[ok]], occ[w, b[ok]] = 0, 1
            E = E + np.where(ok, dE, 0)
            H += np.bincount(E + nb - 1, minlength=nb)
        lnW = _recursion(H, lnW, visited, pacc)
    seen = H[visited]
    return {"H": H, "lnW": lnW, "flat": float(seen.min() / seen.max())}


def _recursion(H, old, visited, pacc):
    """The accumulated-statistics recursion on neighbouring visited energies."""
    visited |= H > 0
    mem = np.nonzero(visited)[0]
    w = old.copy()
    for lo, hi in zip(mem[-2::-1], mem[:0:-1]):
        ratio = old[hi] - old[lo]
        if H[lo] > 0 and H[hi] > 0:
            g = float(H[lo]) * float(H[hi]) / (float(H[lo]) + float(H[hi]))
            pacc[hi] += g
            ratio += g / pacc[hi] * (math.log(H[lo]) - math.log(H[hi]))
        w[lo] = w[hi] - ratio
    above = mem[-1]
    for b in range(len(H) - 1, -1, -1):
        if visited[b]:
            above = b
        else:
            w[b] = old[b] + w[above] - old[above]
    return w - w.max()
