"""The register-tile searches (csrc/hjlo_dense.cuh) where a row's nearest rival
is hardest to see: two sources 4 m apart (one class of the four minima a row
keeps) whose candidates differ by less than the screen's error, at the first
and last rows of lines and row blocks, at segments' first rows and anywhere
else, with the window's end and deeper sources beyond it close by.

On the CPU all four searches (flat; banded with 9 or 13 rows a segment; with 11,
pivots by halving) are written out plainly, one line at a time; a halo entry
past the repeated ones may stand beside a table entry only outside the window.
On the GPU the same lines run through the library.  Both must give the
definition's argmins (every window candidate in binary64, smallest source among
equals)."""
import math

import numpy as np
import pytest

PAD, LOW, HIGH, OVER = 1 << 31, 16, 32, 16
FLAT, WIDE = 4, 11
TOP = 0xffffffff


def _expo(x):
    return math.frexp(x)[1] - 1


def _two(a):
    b = sorted(int(x) for x in a)
    return b[0], b[1]


class Line:
    """One line: lifted[j] = u at halo index j, k[t] = table at offset t; rows
    0 .. NR - 1 are wanted (NR < N: a row block of a periodic line of N)."""

    def __init__(self, u, k, NR, S):
        self.N, self.w, self.NR, self.S = len(u), len(k), NR, S
        self.bits = 7 if S == FLAT else 4 if S == WIDE else 5
        self.mask = (1 << self.bits) - 1
        self.thr = 2 * self.mask + 6
        self.flag = self.thr + self.mask
        N, w = self.N, self.w
        self.u, self.k = np.concatenate([u, u[:w]]), np.asarray(k)
        kmax = float(np.abs(k).max())
        umin, umax = float(u.min()), float(u.max())
        self.q = q = max(_expo((umax - umin + 2 * kmax) * (1 + 2.0 ** -20)) - 30,
                         _expo(max(abs(umin), abs(umax)) + kmax) - 52, -960)
        curv = np.diff(k, 2).min() if w > 2 else math.inf
        assert curv > 2.0 ** (q + self.bits + 3), "the search's condition"
        fix = lambda x: np.trunc(np.asarray(x) / 2.0 ** q).astype(np.int64)     # exact: a power of two
        # the halo repeats the first w entries, then zeros that full bands read
        self.f = np.concatenate([(fix(self.u) - fix(umin)) & ~self.mask, np.zeros(OVER - 1, np.int64)])
        kt = (fix(k) - fix(-kmax)) & ~self.mask
        assert self.f.max() + kt.max() + self.mask < PAD
        self.kt = np.concatenate([np.full(LOW, PAD), kt, np.full(HIGH, PAD)])

    def sums(self, r, js):
        """Screened sums of row r with the sources js, none left out."""
        js = np.asarray(js)
        t = js - r
        assert js.min() >= 0 and js.max() < len(self.f) and t.min() >= -LOW and t.max() < self.w + HIGH
        inside = (t >= 0) & (t < self.w)
        assert not (inside & (js >= self.N + self.w)).any(), "a padding entry as a source"
        return self.f[js] + self.kt[LOW + t]

    def exact(self, r, ts):
        ts = np.asarray(ts)
        return int(ts[np.argmin(self.u[r + ts] + self.k[ts])])

    # ---- the searches: self.lt, self.rows (flagged)
    def run(self):
        self.lt, self.rows = [0] * self.N, set()
        (self.flat if self.S == FLAT else self.banded)()
        N, NR, w, lt = self.N, self.NR, self.w, self.lt
        for r in sorted(self.rows):
            block = NR < N
            lo = r - 1 + lt[r - 1] if r else (0 if block and self.S == FLAT else lt[N - 1] - 1)
            hi = r + 1 + lt[r + 1] if r + 1 < NR else (NR + lt[NR] if block and self.S != FLAT else N + lt[0])
            ts = np.arange(max(lo - r, 0), min(hi - r, w - 1) + 1)
            s = self.sums(r, r + ts)
            near = ts[s <= self.sums(r, [r + lt[r]])[0] + self.thr]
            if len(near) > 1:
                lt[r] = self.exact(r, near)
        return np.array(lt[:NR])

    def flat(self):
        N, NR, w, lt = self.N, self.NR, self.w, self.lt
        nch = (w + 3) >> 2
        kp = np.concatenate([self.kt[LOW:LOW + w] | np.arange(w), np.full(4 * nch - w, PAD)])
        for r in range(NR):
            a = (self.f[r:r + 4 * nch] + kp).reshape(nch, 4).min(0)
            m, m2 = _two(a)
            lt[r] = m & self.mask
            if m2 - m <= self.flag:
                self.rows.add(r)
        for r in range(NR):
            jn = r + 1 + lt[r + 1] if r + 1 < NR else N + lt[0]
            if jn - r - lt[r] >= 4:
                self.rows |= {r, r + 1 if r + 1 < NR else 0}
        if NR < N:
            self.rows.add(0)

    def scan_pivot(self, r):
        """The whole window by one lane: four classes, groups of 4 (mask + 1) displacements."""
        nch, step = (self.w + 3) >> 2, self.mask + 1
        kp = np.full(4 * nch, PAD)
        kp[:self.w] = self.kt[LOW:LOW + self.w]
        kp |= (np.arange(4 * nch) >> 2) & self.mask
        s = (self.f[r:r + 4 * nch] + kp).reshape(nch, 4)
        m = m2 = TOP
        t = 0
        for c0 in range(0, nch, step):
            a = s[c0:c0 + step].min(0)
            b, b2 = _two(a)
            m2 = min(m2, b2, max(m, b))
            if b < m:
                t = 4 * (c0 + (b & self.mask)) + int(np.argmax(a == b))
            m = min(m, b)
        return t, m2 - m <= self.flag

    def pivot_between(self, r, j0, j1):
        """Sources j0 .. j1 of row r by a warp: a true runner-up."""
        js = np.arange(max(j0, r), min(j1, r + self.w - 1) + 1)
        s = self.sums(r, js)
        m, m2 = _two(list(s) + [TOP])
        return int(js[np.argmin(s)]) - r, m2 - m <= self.thr

    def banded(self):
        N, NR, w, S, lt = self.N, self.NR, self.w, self.S, self.lt
        block, nseg = NR < N, -(-NR // S)
        last = lambda: NR + lt[NR] if block else N + lt[0]
        flags = [0] * nseg
        if S == WIDE:
            whole = lambda r: self.pivot_between(r, 0, 1 << 29)
            for g in range(0, nseg, 32):
                lt[g * S], fl = whole(g * S)
                flags[g] |= fl
            if block:
                lt[N - 1], lt[NR] = whole(N - 1)[0], whole(NR)[0]
            for g0 in range(0, nseg, 32):
                d = 16
                while d:
                    for b in range(0, 32, 2 * d):
                        rl = (g0 + b) * S
                        r, rr = rl + d * S, rl + 2 * d * S
                        if r < NR:
                            lt[r], fl = self.pivot_between(r, rl + lt[rl], rr + lt[rr] if rr < NR else last())
                            flags[g0 + b + d] |= fl
                    d >>= 1
        else:
            for g in range(nseg):
                lt[g * S], fl = self.scan_pivot(g * S)
                flags[g] |= fl
            if block:
                lt[N - 1], lt[NR] = self.scan_pivot(N - 1)[0], self.scan_pivot(NR)[0]
                if lt[0] - (lt[N - 1] - 1) >= 4:
                    flags[0] |= 1
        for g in range(nseg):
            s0, s1 = g * S, min(g * S + S, NR)
            jl, jr = s0 + lt[s0], s1 + lt[s1] if s1 < NR else last()
            span = min(jr, s1 + w - 2) - jl + 1
            if span > 16:
                for r in range(s0, s1 + 1):
                    s = self.sums(r, np.arange(jl, jr + 1))
                    m, m2 = _two(list(s) + [TOP])
                    if s0 < r < s1:
                        lt[r] = jl + int(np.argmin(s)) - r
                    if m2 - m <= self.flag and (r < NR or not block):
                        self.rows.add(r if r < NR else 0)
                continue
            jp = jl
            for i in range(1, S + 1):
                j = jr
                if s0 + i < s1:
                    a = (self.sums(s0 + i, np.arange(jl, jl + 16)) + np.arange(16)).reshape(4, 4).min(0)
                    m, m2 = _two(a)
                    j = jl + (m & self.mask)
                    lt[s0 + i] = j - (s0 + i)
                    if m2 - m <= self.flag:
                        flags[g] |= 1 << i
                if j - jp >= 4:
                    flags[g] |= 3 << (i - 1)
                jp = j
        for g in range(nseg):
            s1 = min(g * S + S, NR)
            for b in range(S + 1):
                r = g * S + b
                if flags[g] >> b & 1 and (r < NR or not block):
                    self.rows.add(r if r < NR else 0)


def _table(w, dx, h):
    v = np.arange(w // 2, w // 2 - w, -1, dtype=np.float64) * dx / h
    return h * (0.5 * v * v)


def _rivals(rng, N, k, NR, ends):
    """A line of N points with two sources 4 m apart whose candidates at a row
    r differ by at most 1.5 times the screen's error.  ends: r is the line's
    first row; on a whole line the right source is the window's last."""
    w, curv = len(k), float(k[0] - 2.0 * k[1] + k[2])
    r = 0 if ends else int(rng.choice([0, NR - 1, rng.integers(NR), 9 * rng.integers(-(-NR // 13)) % NR]))
    d = 4 * int(rng.integers(2, min(9, w // 4)))
    right = w - 1 if ends and NR == N else int(rng.integers(d, w))
    u = np.full(N, 400.0 * curv * w) + (rng.random() < 0.5) * curv * rng.normal(size=N)
    unit = 2.0 ** (_expo(float(np.ptp(u)) + 2 * k.max()) - 30)
    at = [(r + right - d) % N, (r + right) % N]
    u[at[0]] = -k[right - d]
    u[at[1]] = -k[right] + rng.uniform(0.0, 100.0) * rng.choice([-1.0, 1.0, 0.0]) * unit
    if rng.random() < 0.7:                       # deeper, just past the row's window
        p = (r + w + int(rng.integers(0, 6))) % N
        if p not in at:
            u[p] = u[at[1]] - rng.uniform(0.0, 40.0) * curv * w
    if rng.random() < 0.3:
        p = (r - int(rng.integers(1, 8))) % N
        if p not in at:
            u[p] = u[at[0]] - rng.uniform(0.0, 40.0) * curv * w
    return u


def _check(u, k, NR, S):
    got = Line(u, k, NR, S).run()
    lifted = np.concatenate([u, u[:len(k) - 1]])
    ref = np.lib.stride_tricks.sliding_window_view(lifted, len(k))[:NR] + k
    return np.array_equal(got, ref.argmin(1)), got - ref.argmin(1)


@pytest.mark.parametrize("ends", [True, False], ids=["ends", "anywhere"])
@pytest.mark.parametrize("block", [False, True], ids=["line", "block"])
@pytest.mark.parametrize("S", [FLAT, 9, 13, WIDE])
def test_close_rivals_are_compared(S, block, ends):
    rng = np.random.default_rng([S, block, ends])
    for n in range(250):
        w = int(rng.integers(40, 97 if S == FLAT else 170))
        NR = int(rng.integers(w, 2 * w)) if block else int(rng.integers(w + 60, 2 * w + 60))
        N = NR + w - 1 if block else NR
        k = _table(w, 1.0 / N, 10 ** rng.uniform(-2.0, -1.3))
        u = _rivals(rng, N, k, NR, ends)
        ok, off = _check(u, k, NR, S)
        assert ok, (n, N, w, NR, np.flatnonzero(off))
