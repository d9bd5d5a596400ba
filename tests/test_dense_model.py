"""The banded monotone search (csrc/hjlo_dense.cuh) written out plainly: keys,
pivots, bands of sources, wide segments and flagged rows, on one line.  Its argmins must equal the definition's (every window candidate in
binary64, smallest source among equals) on smooth fields, shocks, noise, exact
ties and ragged sizes, and every index it forms must lie inside the arrays the
kernel allocates.  Row blocks (fewer rows than points) included."""
import math

import numpy as np
import pytest

PAD, LOW, HIGH, OVER, FLAT = 1 << 31, 16, 32, 16, 4


def _expo(x):
    return math.frexp(x)[1] - 1 if x else -1022


def _fix(x, q):
    """x / 2^q truncated toward zero, exactly."""
    n, d = float(x).as_integer_ratio()
    v = abs(n) * (1 << max(-q, 0)) // (d * (1 << max(q, 0)))
    return v if n >= 0 else -v


def _model(lifted, k, N, NR, S):
    """lifted[jj] = u at halo index jj, k[t] = table at offset t: (argmin offsets,
    statistics).  S: rows per segment, or FLAT: every row over the whole window."""
    bits = 7 if S == FLAT else 5
    MASK = (1 << bits) - 1
    THR = 2 * MASK + 6
    FLAG = THR + MASK
    w = len(k)
    kmax = float(np.abs(k).max())
    umin, umax = float(lifted.min()), float(lifted.max())
    Rk = (umax - umin + 2 * kmax) * (1 + 2.0 ** -20)
    cmax = max(abs(umin), abs(umax)) + kmax
    q = max(_expo(Rk) - 30, _expo(cmax) - 52, -960)
    curv = min((k[t - 1] - 2 * k[t] + k[t + 1] for t in range(1, w - 1)), default=math.inf)
    assert curv > 2.0 ** (q + bits + 3), "the search's condition"
    ref, kref = _fix(umin, q), _fix(-kmax, q)
    f = [(_fix(x, q) - ref) & ~MASK for x in lifted] + [0] * OVER
    kt = [PAD] * LOW + [(_fix(x, q) - kref) & ~MASK for x in k] + [PAD] * HIGH
    kp = [kt[LOW + t] | ((t >> 2) & MASK) for t in range(w)] + [PAD] * (-w % 4)
    assert max(f) + max(x for x in kt if x != PAD) + MASK < PAD

    def F(j):
        assert 0 <= j < N + w - 1 + OVER, j
        return f[j]

    def K(t):
        assert 0 <= t + LOW < len(kt), t
        return kt[t + LOW]

    def exact(r, ts):
        best, bt = math.inf, None
        for t in ts:
            c = lifted[r + t] + k[t]
            if c < best:
                best, bt = c, t
        return bt

    def two(a):
        b = sorted(a)
        return b[0], b[1]

    rows, wide = set(), 0
    nseg, nb = -(-NR // S), 16
    lt = [0] * NR
    flags = [0] * nseg
    if S == FLAT:
        nch = (w + 3) >> 2
        for r0 in range(0, NR, 4):
            for i in range(4):
                a = [0xffffffff] * 4
                for c in range(nch):
                    for e in range(4):
                        t = 4 * c + e
                        a[e] = min(a[e], F(r0 + i + t) + (kt[LOW + t] | t if t < w else PAD))
                if r0 + i < NR:
                    m, m2 = two(a)
                    lt[r0 + i] = m & MASK
                    if m2 - m <= FLAG:
                        rows.add(r0 + i)
            F(r0 + 4 * nch + 3)
        for r in range(NR):
            jn = r + 1 + lt[r + 1] if r + 1 < NR else N + lt[0]
            if jn - r - lt[r] >= 4:
                rows |= {r, (r + 1) if r + 1 < NR else 0}
        if NR < N:
            rows.add(0)
        nseg = 0
    outer = [NR, N - 1] if NR < N and S != FLAT else []    # the rows after and before a row block
    lt += [0] * (N - NR)
    for g in range(nseg + len(outer)):
        s0, m, m2, t = (g * S if g < nseg else outer[g - nseg]), 0xffffffff, 0xffffffff, 0
        nch = (w + 3) >> 2
        for c0 in range(0, nch, 32):
            a = [0xffffffff] * 4
            for c in range(c0, min(c0 + 32, nch)):
                for e in range(4):
                    a[e] = min(a[e], F(s0 + 4 * c + e) + kp[4 * c + e])
            b, b2 = two(a)
            tb = 4 * (c0 + (b & MASK)) + a.index(b)
            m2 = min(m2, b2, max(m, b))
            t = tb if b < m else t
            m = min(m, b)
        lt[s0] = t
        if g < nseg and m2 - m <= FLAG:
            flags[g] |= 1

    def last():
        return NR + lt[NR] if NR < N else N + lt[0]

    for g in range(nseg):
        s0, s1 = g * S, min(g * S + S, NR)
        jl = s0 + lt[s0]
        jr = s1 + lt[s1] if s1 < NR else last()
        jc = min(jr, s1 + w - 2)
        span = jc - jl + 1
        assert span >= 1
        if span > nb:
            wide += 1
            for i in range(s1 - s0 + 1):
                r = s0 + i
                js = list(range(jl, jr + 1))
                keys = [F(j) + K(j - r) for j in js]
                b, b2 = two(keys + [0xffffffff])
                if 0 < i < S and r < NR:
                    lt[r] = js[keys.index(b)] - r
                if b2 - b <= FLAG and (r < NR or NR == N):
                    rows.add(r if r < NR else 0)
            continue
        acc = [[0xffffffff] * 4 for _ in range(S - 1)]
        for c in range(nb // 4):                         # a full band, as the widest bracket of a warp asks for
            for e in range(4):
                for i in range(1, S):
                    v = F(jl + 4 * c + e) + 4 * c + e + K(jl - s0 + 4 * c + e - i)
                    acc[i - 1][e] = min(acc[i - 1][e], v)
        jp = jl
        for i in range(1, S + 1):
            j = jr
            if i < S and s0 + i < s1:
                m, m2 = two(acc[i - 1])
                j = jl + (m & MASK)
                lt[s0 + i] = j - (s0 + i)
                if m2 - m <= FLAG:
                    flags[g] |= 1 << i
            if j - jp >= 4:
                flags[g] |= 3 << (i - 1)
            jp = j
    for g in range(nseg):
        s0, s1 = g * S, min(g * S + S, NR)
        for b in range(S + 1):
            if flags[g] >> b & 1:
                r = s0 + b
                if r < NR or NR == N:
                    rows.add(r if r < s1 else (s1 if s1 < NR else 0))
    for r in sorted(rows):
        lo = r - 1 + lt[r - 1] if r else (0 if S == FLAT and NR < N else lt[N - 1] - 1)
        hi = r + 1 + lt[r + 1] if r + 1 < NR else (last() if S != FLAT else N + lt[0])
        ts = range(max(lo - r, 0), min(hi - r, w - 1) + 1)
        m = F(r + lt[r]) + K(lt[r])
        near = [t for t in ts if F(r + t) + K(t) <= m + THR]
        if len(near) > 1:
            lt[r] = exact(r, near)
    return lt, dict(flagged=len(rows), wide=wide)


def _field(kind, n, rng, a):
    x = np.arange(n) / n
    if kind == "shocks":
        fs = [rng.normal() * 0.3 * np.cos(2 * np.pi * (x * rng.integers(1, 4) + rng.random())) for _ in range(6)]
        u = np.min(fs, axis=0)
        return u - 0.5 * np.abs(np.sin(np.pi * (3 * x + rng.random())))
    if kind == "noise":
        return rng.normal(size=n) * 0.3
    if kind == "wells":                               # sources 25 apart, every other one best on 3 rows only
        u = np.full(n, 2000.0 * a)
        u[::50] = 0.0
        u[25::50] = 275.0 * a
        return u
    if kind == "ties":
        return rng.integers(0, 3, size=n) / 8.0
    if kind == "flat":
        return np.zeros(n)
    return 40.0 + 0.3 * np.sin(2 * np.pi * x + rng.random())      # far from zero


@pytest.mark.parametrize("kind", ["shocks", "noise", "wells", "ties", "flat", "offset"])
@pytest.mark.parametrize("S", [FLAT, 9, 13])
def test_banded_search_finds_the_argmins(kind, S):
    rng = np.random.default_rng([S, len(kind)])
    seen = dict(flagged=0, wide=0)
    for N, weff in [(1, 1), (2, 2), (5, 3), (9, 9), (10, 4), (27, 7), (64, 65 - 2), (101, 33), (130, 129), (150, 65),
                    (260, 131)]:
        weff = min(weff, N, 96 if S == FLAT else N)
        for NR in {N, N - weff + 1}:                  # whole lines, and a block's own rows
            dx, h, P = 1.0 / N, float(rng.uniform(0.01, 0.1)), float(rng.choice([0.0, 0.5 * N ** -1, 0.7]))
            c = round(P * h / dx)
            d = np.arange(c + weff // 2, c + weff // 2 - weff, -1, dtype=np.float64)
            v = d * dx / h
            k = h * (0.5 * v * v - P * v)
            u = _field(kind, N, rng, dx * dx / h)
            lifted = np.concatenate([u, u[:weff - 1]])
            got, n = _model(lifted, k, N, NR, S)
            for r in range(NR):
                cand = lifted[r:r + weff] + k
                assert got[r] == int(np.argmin(cand)), (N, weff, NR, r)
            seen = {q: seen[q] + n[q] for q in seen}
    if kind == "wells":
        assert seen["flagged"] > 0 and (seen["wide"] > 0 or S == FLAT)        # every path was taken


@pytest.mark.parametrize("S", [FLAT, 9, 13])
def test_banded_search_on_rough_lines(S):
    """Random lines, windows, steps and roughness: brackets with and without gaps of every length."""
    rng = np.random.default_rng([S, 77])
    done = 0
    while done < 150:
        N = int(rng.integers(20, 300))
        weff = min(N, int(rng.integers(20, 97 if S == FLAT else 160)))
        NR = int(rng.choice([N, N - weff + 1]))
        h, dx = 10 ** rng.uniform(-3, -1), 1.0 / N
        x = np.arange(N) / N
        u = 0.3 * rng.random() * np.sin(2 * np.pi * (x + rng.random())) + 10 ** rng.uniform(-4, 0) * rng.normal(size=N)
        v = np.arange(weff // 2, weff // 2 - weff, -1, dtype=np.float64) * dx / h
        k = h * (0.5 * v * v)
        lifted = np.concatenate([u, u[:weff - 1]])
        if not 0.9 * dx * dx / h > 2.0 ** (_expo(float(np.ptp(u)) + 2 * k.max()) - (18 if S == FLAT else 20)):
            continue                                  # curvature too small for the bands
        got, _ = _model(lifted, k, N, NR, S)
        done += 1
        for r in range(NR):
            assert got[r] == int(np.argmin(lifted[r:r + weff] + k)), (N, weff, NR, r)
