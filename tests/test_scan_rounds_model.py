"""The rounds with several commits (walker_scan.cuh), restated lane by lane in
plain Python: the sliding window of attempts, the recurrence in the energy, the
pairwise tests for touching around the ring of slots, rounds up to the first
accepted attempt, and the three sources of thresholds.  The model reproduces
the serial chain, and a wait for threshold rows that runs out in some lanes of
a group only still ends the rounds."""
import os
import re

import numpy as np
import pytest

from oracle import chain

PAD, WORDS, REACH, ROWS, DRIFT = 16, 24, 10, 32, 9
WLO, WHI = ROWS // 2 - 1, ROWS // 2


class Endless(Exception):
    pass


class Wait:
    """Outcomes of the lanes' waits: lane l's n-th wait runs out if (l, n) is listed."""

    def __init__(self, out=(), vote=True):
        self.out, self.vote, self.n = set(out), vote, 0

    def __call__(self, broken):
        got = [b or (l, self.n) in self.out for l, b in enumerate(broken)]
        self.n += 1
        return [any(got)] * len(got) if self.vote else got


def serial(d, L, N, S, occ, x, T, att):
    H = np.zeros(T.shape[0], np.int64)
    for k, m, r in att:
        a, b = int(S[k]), int(S[N + m])
        j = chain.delta_e(d, L, occ, a, b) + 2 * d
        if int(T[x, j]) >= r:
            occ[a], occ[b] = 0, 1
            S[k], S[N + m] = b, a
            x += j - 2 * d
        H[x] += 1
    return x, H


def rounds(d, L, N, S, occ, x, T, att, A, W, mode, rng, wait, others=0.0):
    """One walker's group of W lanes over A attempts; `others` is the chance
    that another walker of the warp had many accepted moves.  Returns the
    energy bin, the histogram, whether a wait ran out, and the rounds taken."""
    nb, dead, few = T.shape[0], 4 * d + 1, W // 4
    H = np.zeros(nb, np.int64)
    lanes = range(W)
    garbage = lambda: int(rng.integers(1 << 32))                      # noqa: E731
    ring = [None] * ROWS                                              # row that has arrived in a slot
    c, flying, vlo, vhi = x, [], [x - WLO] * W, [x + WHI] * W
    t0, broken, bin_, carry, many = [0] * W, [False] * W, x, 0, True

    def fetch(r0, r1):
        r0, r1 = max(r0, 0), min(r1, nb - 1)
        for r in range(r0, r1 + 1):
            ring[r % ROWS] = None
        flying.extend(range(r0, r1 + 1))

    def land():
        nonlocal broken
        if flying and not all(broken):
            broken = wait(broken)
            for r in flying:
                ring[r % ROWS] = r
            flying.clear()

    def row(y, code):
        if code == dead:
            return 0 if 0 <= y < nb and (mode != "window" or ring[y % ROWS] == y) else garbage()
        if mode == "window" and ring[y % ROWS] != y:
            return garbage()
        return int(T[y, code])

    if mode == "window":
        fetch(x - WLO, x + WHI)
        land()
    cur = list(att[:W])
    a, b = [int(S[q[0]]) for q in cur], [int(S[N + q[1]]) for q in cur]
    n_rounds = 0
    while any(t < A for t in t0) and not all(broken):
        n_rounds += 1
        if n_rounds > 4 * A + 16:
            raise Endless
        if mode == "window":
            if flying:
                land()
                vlo, vhi = [c - WLO] * W, [c + WHI] * W
            if not all(broken) and abs(bin_ - c) > DRIFT:
                if bin_ > c:
                    fetch(max(c + WHI + 1, bin_ - WLO), bin_ + WHI)
                else:
                    fetch(bin_ - WLO, min(c - WLO - 1, bin_ + WHI))
                vlo, vhi = [max(v, bin_ - WLO) for v in vlo], [min(v, bin_ + WHI) for v in vhi]
                c = bin_
                if flying and not vlo[0] <= bin_ <= vhi[0]:
                    land()
                if not flying:
                    vlo, vhi = [c - WLO] * W, [c + WHI] * W
            t0 = [A if broken[l] else t0[l] for l in lanes]
        near = [min(max(A - t, 0), 3 * W) for t in t0]
        place = [(l - t0[l]) % W for l in lanes]
        nxt = [att[t0[l] + place[l] + W] if t0[l] < A else cur[l] for l in lanes]
        an, bn = [int(S[q[0]]) for q in nxt], [int(S[N + q[1]]) for q in nxt]
        code = [chain.delta_e(d, L, occ, a[l], b[l]) + 2 * d if place[l] < near[l] else dead for l in lanes]
        nv = [min(n, W) for n in near]
        at = {place[l]: l for l in lanes}
        if len(at) < W:                                                # lanes of different attempts
            decided = []
        elif not many:
            yes = [l for l in lanes if place[l] < nv[l] and row(bin_, code[l]) >= cur[l][2]]
            first = min((place[l] for l in yes), default=None)
            nd = nv[0] if first is None else first + 1
            many = len(yes) > few
            decided = [l for l in lanes if place[l] < nd]
            commits = [] if first is None else [at[first]]
            after = [bin_] * nd
            if commits:
                after[-1] += code[commits[0]] - 2 * d
        else:
            e0 = (bin_ + PAD - REACH) & ~3
            y, accepted, xs, valid = bin_, [], [], []
            for i in range(W):
                l = at[i]
                if mode == "global":
                    ok = 0
                    for q in range(WORDS):
                        r = e0 + q - PAD
                        t = int(T[r, code[l]]) if 0 <= r < nb and code[l] != dead else 0
                        ok |= (t >= cur[l][2] and code[l] != dead) << q
                    s = y + PAD - e0
                    take = (code[l] << 24 | ok) >> (s % 32) & 1
                    valid.append(0 <= s < WORDS)
                else:
                    take = row(y, code[l]) >= cur[l][2]
                    valid.append(mode == "shared" or vlo[0] <= y <= vhi[0])
                y += code[l] - 2 * d if take else 0
                accepted.append(bool(take) and i < nv[0])
                xs.append(y)
            around = [set(chain.neighbours(d, L, a[l]).tolist()) | set(chain.neighbours(d, L, b[l]).tolist())
                      for l in lanes]
            bad = {i for i in range(W) if not valid[i]}
            for l in lanes:
                for q in range(1, W // 2 + 1):                         # the W / 2 slots behind it in the ring
                    o = (l + q) % W
                    if a[o] in around[l] or b[o] in around[l] or a[o] == a[l] or b[o] == b[l]:
                        i, e = place[l], place[o]
                        if accepted[min(i, e)]:
                            bad.add(max(i, e))
            nd = min(bad | {nv[0]})
            many = sum(accepted) > few
            decided = [l for l in lanes if place[l] < nd]
            commits = [l for l in decided if accepted[place[l]]]
            after = xs[:nd]
        many = many or rng.random() < others
        if not decided:
            continue
        for e in after:                          # runs of one energy, added when it changes
            if e == bin_:
                carry += 1
            else:
                H[bin_] += carry
                bin_, carry = e, 1
        for l in commits:
            k, m, _ = cur[l]
            occ[a[l]], occ[b[l]] = 0, 1
            S[k], S[N + m] = b[l], a[l]
        moved = [(cur[l][0], cur[l][1], a[l], b[l]) for l in commits]
        for l in decided:
            cur[l], a[l], b[l] = nxt[l], an[l], bn[l]
        for k, m, pa, pb in moved:               # list entries read before the commits
            for l in lanes:
                a[l] = pb if cur[l][0] == k else a[l]
                b[l] = pa if cur[l][1] == m else b[l]
        t0 = [t + len(decided) for t in t0]
    H[bin_] += carry
    return bin_, H, any(broken), n_rounds


def _walker(d, L, N, slope, noise):
    rng = np.random.default_rng(100 * d + 10 * L + N)
    nb = d * N + 1
    T = chain.thresholds(d, -d * N, 0, slope * np.arange(nb) + noise * rng.standard_normal(nb))
    S, occ, E = chain.init_walkers(d, L, N, 1, 7 + N)
    return rng, T, S[0], occ[0], int(E[0]) + d * N


def _attempts(rng, L, d, N, n):
    r = rng.integers(1 << 32, size=n, dtype=np.int64)
    r = np.where(r == 0xFFFFFFFF, r, r + 1)       # T >= r accepts
    return list(zip(rng.integers(N, size=n).tolist(), rng.integers(L ** d - N, size=n).tolist(), r.tolist()))


@pytest.mark.parametrize("mode", ["shared", "window", "global"])
@pytest.mark.parametrize("d,L,N,W,slope,noise", [
    (2, 6, 9, 4, 0.0, 0.0), (2, 9, 30, 8, -0.8, 0.3), (2, 3, 4, 8, 0.0, 0.5), (2, 12, 60, 32, 0.3, 0.1),
    (3, 3, 13, 4, 0.0, 0.6), (3, 6, 60, 16, -1.5, 0.2), (3, 5, 60, 8, 0.0, 0.0), (2, 6, 35, 4, 0.0, 0.0)])
def test_rounds_are_the_serial_chain(d, L, N, W, slope, noise, mode):
    rng, T, S, occ, x = _walker(d, L, N, slope, noise)
    S0, occ0, x0 = S.copy(), occ.copy(), x
    for A, others in ((1, 0.0), (W - 1, 0.0), (613, 0.0), (401, 0.5)):
        att = _attempts(rng, L, d, N, A + 3 * W)
        x0, H0 = serial(d, L, N, S0, occ0, x0, T, att[:A])
        x, H, broken, _ = rounds(d, L, N, S, occ, x, T, att, A, W, mode, rng, Wait(), others)
        assert x == x0 and not broken
        np.testing.assert_array_equal(H, H0)
        np.testing.assert_array_equal(S, S0)
        np.testing.assert_array_equal(occ, occ0)


def test_a_wait_that_runs_out_ends_the_rounds():
    """Lanes that do not share the outcome can keep the rounds going for ever."""
    def run(out, vote):
        rng, T, S, occ, x = _walker(2, 14, 80, -0.8, 0.0)
        wait = Wait(out, vote)
        rounds(2, 14, 80, S, occ, x, T, _attempts(rng, 14, 2, 80, 924), 900, 8, "window", rng, wait)
        return wait.n
    waits = run((), True)
    assert waits >= 3
    for n in range(waits):
        for out in ([0], [5], list(range(7)), list(range(8))):
            run([(l, n) for l in out], True)
    with pytest.raises(Endless):
        run([(5, 1)], False)
    # the rounds have no wait whose outcome is a lane's own
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1401_4076_gb300", "csrc",
                        "walker_scan.cuh")
    with open(path) as f:
        calls = re.findall(r"tw\.(wait\w*)\(([^)]*)\)", f.read())
    assert calls and set(calls) == {("wait_group", "p, gm")}
