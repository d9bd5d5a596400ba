"""Workload cases of the Lax--Oleinik solver, for timing and for checking.

Each case is one call (or one run of calls) a user's program makes through the
public Python binding: `prepare` builds what such a program holds (device
fields, a plan or a batch), `run` makes the call and returns its whole result,
`work` counts the bytes and operations the result needs, and `exact` gives the
result from the definition in binary64 with plain torch operations.

Kinds of case:
  run       n steps of a 1D/2D/3D grid in place (Plan.run), from a stored state
  step      one step with its argmins (Plan.step)
  run_tv    n steps with a potential per step (Plan.run_tv)
  batch     many 2D grids advanced together and their H-bar (Batch.run, .hbar)
  adjoint   gradients of n steps w.r.t. u0, P and V (Plan.adjoint)
  decomp    n steps by the decomposition method at tolerance eta = dx
  integral  n steps of the first discrete semigroup (IntegralPlan.run)

Grids are unit tori (dx = 1/N per axis, h = 0.02) except the 1D lines of the
pendulum law on (0, 2 pi] with tau = T/ceil(T/sqrt(dx)).  A stored state is a
minimum of smooth functions: solutions of the scheme are semiconcave, smooth
between the shocks where two branches cross.
"""
import math

import numpy as np
import torch

from paper_1210_4090_gb300 import hjlo

_H = 0.02


def listed():
    return [
        # one short line, every candidate of the torus window: the smallest
        # problem, where each step is bound by its launch
        dict(name="line256", kind="run", law="torus", n0=256, n1=0, n2=0, W=0, steps=200, f32=False, algo="brute"),
        # a program that looks at the solution and its optimal paths after every step
        dict(name="step128_argmin", kind="step", n0=128, n1=128, W=8, f32=False),
        # the 2D run of the benchmark set
        dict(name="grid1024", kind="run", law="torus", n0=1024, n1=1024, n2=0, W=64, steps=64, f32=False,
             algo="auto"),
        # 2D with ragged sizes and 32-bit storage
        dict(name="grid_odd_f32", kind="run", law="torus", n0=701, n1=1013, n2=0, W=63, steps=48, f32=True,
             algo="auto"),
        # the 3D run of the benchmark set, its fields larger than L2
        dict(name="cube256", kind="run", law="torus", n0=256, n1=256, n2=256, W=32, steps=16, f32=False,
             algo="auto"),
        # 3D with ragged sizes
        dict(name="cube_odd", kind="run", law="torus", n0=90, n1=121, n2=135, W=12, steps=24, f32=False,
             algo="auto"),
        # a sweep of the effective Hamiltonian over P on mixed grid sizes
        dict(name="sweep40", kind="batch", count=40, nlo=128, nhi=512, steps=32, f32=False),
        # gradients for fitting P and V
        dict(name="adjoint512", kind="adjoint", n0=512, n1=512, W=32, steps=128, every=32),
        # the first quarter of the pendulum run on 2^18 points, one long line
        dict(name="pendulum_2p18", kind="run", law="pendulum", n0=1 << 18, n1=0, n2=0, W=1635, steps=400, f32=False,
             algo="auto"),
        # the time-dependent potential on 2 x 4096 points
        dict(name="tdep_8192", kind="run_tv", n0=8192, steps=289),
        # the whole pendulum run on 2^18 points by the decomposition method
        dict(name="decomp_2p18", kind="decomp", n0=1 << 18, steps=1635),
        # the first discrete semigroup
        dict(name="integral128", kind="integral", n0=128, n1=128, W=4, modes=2, steps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "step", "run_tv", "batch", "adjoint", "decomp", "integral"])
    if kind == "run":
        nd = rng.choice([1, 2, 2, 3, 3])
        f32 = rng.random() < 0.3
        if nd == 1 and rng.random() < 0.5:
            n = _log(rng, 64, 2048)
            return dict(kind="run", law="torus", n0=n, n1=0, n2=0, W=rng.choice([0, max(4, n // 12)]),
                        steps=rng.randint(20, 200), f32=f32, algo=rng.choice(["auto", "brute"]))
        if nd == 1:
            n = 2 * _log(rng, 1 << 11, 1 << 17)
            W = int(math.ceil(4.0 * _pendulum_step(n)[1] / _pendulum_step(n)[0])) + 1
            return dict(kind="run", law="pendulum", n0=n, n1=0, n2=0, W=W, steps=rng.randint(40, 200), f32=f32,
                        algo="auto")
        if nd == 2:
            n = [_log(rng, 96, 1024) for _ in range(2)]
            most = (64 << 20) // (n[0] * n[1])
            return dict(kind="run", law="torus", n0=n[0], n1=n[1], n2=0,
                        W=_log(rng, max(4, max(n) // 20), max(5, max(n) // 8)),
                        steps=rng.randint(4, max(4, min(128, most))), f32=f32, algo="auto")
        n = [_log(rng, 24, 256) for _ in range(3)]
        most = (16 << 24) // (n[0] * n[1] * n[2])
        return dict(kind="run", law="torus", n0=n[0], n1=n[1], n2=n[2],
                    W=_log(rng, max(4, max(n) // 16), max(5, max(n) // 8)),
                    steps=rng.randint(4, max(4, min(64, most))), f32=f32, algo="auto")
    if kind == "step":
        n = [_log(rng, 32, 1024) for _ in range(2)]
        return dict(kind="step", n0=n[0], n1=n[1], W=_log(rng, max(3, max(n) // 20), max(4, max(n) // 8)),
                    f32=rng.random() < 0.3)
    if kind == "run_tv":
        n = 2 * _log(rng, 64, 8192)
        return dict(kind="run_tv", n0=n, steps=rng.randint(20, 300))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 40), nlo=64 * rng.randint(1, 3), nhi=64 * rng.randint(4, 8),
                    steps=rng.randint(4, 32), f32=rng.random() < 0.3)
    if kind == "adjoint":
        n = [_log(rng, 64, 512) for _ in range(2)]
        return dict(kind="adjoint", n0=n[0], n1=n[1], W=_log(rng, max(4, max(n) // 20), max(5, max(n) // 8)),
                    steps=rng.randint(16, 128), every=rng.choice([0, 8, 20, 32]))
    if kind == "decomp":
        n = 2 * _log(rng, 1 << 11, 1 << 17)
        return dict(kind="decomp", n0=n, steps=rng.randint(50, 1000))
    n = [_log(rng, 32, 128) for _ in range(2)]
    return dict(kind="integral", n0=n[0], n1=n[1], W=rng.randint(2, 4), modes=rng.randint(1, 2),
                steps=rng.randint(2, 16))


# ---------------------------------------------------------------- inputs

def _shape(case):
    return tuple(case[k] for k in ("n0", "n1", "n2") if case.get(k))


def _modes(ndim, K):
    """Integer modes 0 < |k|_inf <= K, one of each +-k pair."""
    ks = np.array(list(np.ndindex(*([2 * K + 1] * ndim))), dtype=np.int64) - K
    keep = [k for k in ks if k.any() and k[np.flatnonzero(k)[0]] > 0]
    return np.array(keep, dtype=np.int64).reshape(-1, ndim)


def _series(shape, modes, coef):
    """sum_m Re(coef_m exp(2 pi i k_m . x)) at x_a = i_a / shape[a], on the GPU."""
    nd, K = len(shape), int(np.abs(modes).max())
    C = np.zeros([2 * K + 1] * nd, dtype=np.complex128)
    for k, c in zip(modes, coef):
        C[tuple(int(x) + K for x in k)] += c
    out = torch.tensor(C, device="cuda")
    ks = torch.arange(-K, K + 1, dtype=torch.float64, device="cuda")
    for n in shape:
        t = 2.0 * math.pi * torch.outer(ks, torch.arange(n, dtype=torch.float64, device="cuda") / n)
        out = torch.tensordot(out, torch.complex(torch.cos(t), torch.sin(t)), dims=([0], [0]))
    return out.real.contiguous()


def _gauss(rng, shape, K, var):
    """Random real Fourier series, cos and sin coefficients ~ N(0, var / |k|^2)."""
    m = _modes(len(shape), K)
    s = math.sqrt(var) / np.sqrt((m.astype(np.float64) ** 2).sum(1))
    return _series(shape, m, rng.normal(size=len(m)) * s - 1j * rng.normal(size=len(m)) * s)


def _state(rng, shape):
    """A minimum of four smooth fields with slopes of about 2."""
    m = _modes(len(shape), 2)
    u = None
    for _ in range(4):
        c = (rng.normal(size=len(m)) + 1j * rng.normal(size=len(m))) / np.sqrt((m.astype(np.float64) ** 2).sum(1))
        c *= 2.0 / (2.0 * math.pi * math.sqrt(len(m)))
        f = _series(shape, m, c)
        u = f if u is None else torch.minimum(u, f)
    return u


def _pendulum_step(n, T=8.0):
    dx = 2.0 * math.pi / n
    return dx, T / math.ceil(T / math.sqrt(dx) - 1e-12)


def _problem(case, seed):
    """The case's geometry and its device fields: dict(shape, dx, h, P, W, u0, V)."""
    rng = np.random.default_rng([int(seed), 1210])
    kind = case["kind"]
    if kind in ("run_tv", "decomp") or case.get("law") == "pendulum":
        n = case["n0"]
        dx, tau = _pendulum_step(n)
        W = case.get("W") or int(math.ceil(4.0 * tau / dx)) + 1
        W = 0 if 2 * W + 1 >= n else W
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 1.0) * dx
        amp, phase, shift = rng.uniform(0.8, 1.2), rng.uniform(0, 2 * math.pi), rng.uniform(-0.3, 0.3)
        u0 = torch.cos(x + phase)
        if kind == "run_tv":
            t = torch.arange(case["steps"], dtype=torch.float64, device="cuda") * tau
            V = amp * torch.sin(t + shift)[:, None] * torch.cos(2.0 * x + 2.0 * phase)[None, :]
            return dict(shape=(n,), dx=(dx,), h=tau, P=(1.0,), W=(W,), u0=u0, V=V.contiguous())
        V = amp * (1.0 - torch.cos(x + phase + shift))
        return dict(shape=(n,), dx=(dx,), h=tau, P=(0.0,), W=(W,), u0=u0, V=V)
    shape = _shape(case)
    nd = len(shape)
    P = tuple(float(p) for p in rng.uniform(-0.4, 0.4, nd))
    dx = tuple(1.0 / n for n in shape)
    if nd == 1:
        V, h = _gauss(rng, shape, 4, 0.05), 0.05
    else:
        V, h = _gauss(rng, shape, 6 if nd == 2 else 4, 0.25 if nd == 2 else 0.2), _H
    return dict(shape=shape, dx=dx, h=h, P=P, W=(case["W"],) * nd, u0=_state(rng, shape), V=V)


def _batch_sizes(case):
    """Grid sizes of a batch, nlo..nhi in steps of 64 (they do not depend on the seed)."""
    sizes = np.arange(case["nlo"], case["nhi"] + 1, 64)
    return [int(np.random.default_rng([case["count"], i]).choice(sizes)) for i in range(case["count"])]


def _instances(case, seed):
    """The grids of a batch: P over [-1, 1]^2, W = N/16."""
    out = []
    for i, N in enumerate(_batch_sizes(case)):
        rng = np.random.default_rng([int(seed), 1210, i])
        P = tuple(float(p) for p in rng.uniform(-1.0, 1.0, 2))
        m = _modes(2, 4)
        amp = rng.uniform(-0.5, 0.5, len(m)) / np.sqrt((m.astype(np.float64) ** 2).sum(1))
        V = _series((N, N), m, amp * np.exp(1j * rng.uniform(0, 2 * math.pi, len(m))))
        out.append(dict(shape=(N, N), dx=(1.0 / N,) * 2, h=_H, P=P, W=(N // 16,) * 2, V=V,
                        u0=_state(rng, (N, N))))
    return out


def _cotangent(shape, seed):
    """Weights of a weighted mean of u^n: a smooth field about 1."""
    return 1.0 + _gauss(np.random.default_rng([int(seed), 4090]), shape, 3, 0.05)


def _integral_terms(case, seed):
    rng = np.random.default_rng([int(seed), 1210])
    shape = _shape(case)
    m = _modes(2, case["modes"])
    s = 0.5 / np.sqrt((m.astype(np.float64) ** 2).sum(1))
    coef = rng.normal(size=len(m)) * s - 1j * rng.normal(size=len(m)) * s
    P = tuple(float(p) for p in rng.uniform(-0.4, 0.4, 2))
    return dict(shape=shape, dx=tuple(1.0 / n for n in shape), h=_H, P=P, W=(case["W"],) * 2, modes=m, coef=coef,
                u0=_state(rng, shape))


# ---------------------------------------------------------------- the calls

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ps = _instances(case, seed)
        typ = torch.float32 if case["f32"] else torch.float64
        batch = hjlo.Batch([(p["shape"], p["dx"], p["h"], p["P"], p["W"]) for p in ps],
                           dtype=hjlo.F32_STORAGE if case["f32"] else hjlo.F64)
        u0 = [p["u0"].to(typ) for p in ps]
        return dict(case=case, batch=batch, u0=u0, u=[torch.empty_like(x) for x in u0], V=[p["V"] for p in ps])
    if kind == "integral":
        p = _integral_terms(case, seed)
        plan = hjlo.IntegralPlan(p["shape"], p["dx"], p["h"], p["P"], p["W"], p["modes"], p["coef"])
        return dict(case=case, plan=plan, u0=p["u0"], u=torch.empty_like(p["u0"]))
    p = _problem(case, seed)
    f32 = bool(case.get("f32"))
    algo = {"brute": hjlo.ALGO_BRUTE}.get(case.get("algo"), hjlo.ALGO_AUTO)
    plan = hjlo.Plan(p["shape"], p["dx"], p["h"], p["P"], p["W"], dtype=hjlo.F32_STORAGE if f32 else hjlo.F64,
                     algo=hjlo.ALGO_DECOMP if kind == "decomp" else algo)
    if kind == "decomp":
        plan.set_tolerance(p["dx"][0])
    u0 = p["u0"].to(torch.float32) if f32 else p["u0"]
    s = dict(case=case, plan=plan, u0=u0, u=torch.empty_like(u0), V=p["V"])
    if kind == "step":
        s["argmin"] = torch.empty((2,) + p["shape"], dtype=torch.int32, device="cuda")
    if kind == "adjoint":
        s["ubar"] = _cotangent(p["shape"], seed)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        u = state["plan"].step(state["u0"], state["u"], state["V"], argmin=state["argmin"])
        return {"u": u, "argmin": state["argmin"]}
    if kind == "adjoint":
        ubar0, Pbar, Vbar, un = state["plan"].adjoint(state["u0"], state["V"], case["steps"], state["ubar"],
                                                      checkpoint_every=case["every"], want_un=True)
        return {"ubar0": ubar0, "Pbar": Pbar, "Vbar": Vbar, "un": un}
    if kind == "batch":
        for u, u0 in zip(state["u"], state["u0"]):
            u.copy_(u0)
        state["batch"].run(state["u"], state["V"], case["steps"])
        return {"u": list(state["u"]), "hbar": state["batch"].hbar(state["u0"], state["u"], case["steps"])}
    u = state["u"]
    u.copy_(state["u0"])
    if kind == "integral":
        return state["plan"].run(u, case["steps"])
    if kind == "run_tv":
        return state["plan"].run_tv(u, state["V"], case["steps"])
    return state["plan"].run(u, state["V"], case["steps"])


# ---------------------------------------------------------------- what a pass needs

def work(case):
    """Bytes: every input read once, every output written once.  Operations:
    one binary64 add per output and axis, and the potential term, per step (the
    integral semigroup evaluates its whole box: a multiply and an add per mode
    component and four more per candidate)."""
    kind = case["kind"]
    if kind == "batch":
        pts = sum(N * N for N in _batch_sizes(case))
        e = 4 if case["f32"] else 8
        return {"bytes": pts * (2 * e + 8), "flops": 3 * pts * case["steps"]}
    pts, nd = int(np.prod(_shape(case))), len(_shape(case))
    e = 4 if case.get("f32") else 8
    steps = case.get("steps", 1)
    if kind == "integral":
        box = (2 * case["W"] + 1) ** 2
        modes = ((2 * case["modes"] + 1) ** 2 - 1) // 2
        return {"bytes": pts * 16, "flops": pts * steps * box * (4 * modes + 4)}
    if kind == "adjoint":
        # forward, and its transpose: one add per routed cotangent and axis,
        # the two products' sums for P and the potential's
        return {"bytes": pts * 8 * 6, "flops": pts * steps * ((nd + 1) + (3 * nd + 2))}
    if kind == "run_tv":
        return {"bytes": pts * (16 + 8 * steps), "flops": pts * steps * (nd + 2)}
    extra = 4 * nd * pts if kind == "step" else 0
    return {"bytes": pts * (2 * e + 8) + extra, "flops": pts * steps * (nd + 1)}


# ---------------------------------------------------------------- the definition in binary64

def _window(N, dx, h, P, W):
    """Displacements (ascending) and kernel values k[d] = h (v^2/2 - P v), v = d dx / h."""
    def k(d):
        v = (d * dx) / h
        return h * ((0.5 * v) * v - P * v)
    base = math.floor(P * h / dx)
    c = max(range(base - 5, base + 7), key=lambda d: (-k(d), d))
    if 0 < W and 2 * W + 1 < N:
        lo, hi = c - W, c + W
    else:
        lo = hi = c
        while hi - lo + 1 < N:
            if k(lo - 1) < k(hi + 1):
                lo -= 1
            else:
                hi += 1
    return lo, [k(d) for d in range(lo, hi + 1)]


def _axis_min(u, axis, lo, k):
    """min_d u[(i - d) mod N] + k[d] along an axis."""
    N, w = u.shape[axis], len(k)
    if u.dim() == 1 and w > 64:
        # rows of the lifted window: u[(i - d) mod N], d descending
        hi = lo + w - 1
        idx = (torch.arange(N + w - 1, device=u.device) - hi) % N
        lifted = u[idx]
        kr = torch.tensor(k[::-1], dtype=torch.float64, device=u.device)
        rows = max(1, (1 << 28) // w)
        return torch.cat([(lifted.as_strided((min(rows, N - r), w), (1, 1), r) + kr).amin(1)
                          for r in range(0, N, rows)])
    m = None
    for t, kd in enumerate(k):
        c = torch.roll(u, lo + t, axis) + kd
        m = c if m is None else torch.minimum(m, c)
    return m


def _axis_argmin(u, axis, lo, k):
    """The pass and its argmin displacement (smallest lifted source, i.e. largest d, among equals)."""
    m = torch.roll(u, lo + len(k) - 1, axis) + k[-1]
    a = torch.full(u.shape, lo + len(k) - 1, dtype=torch.int64, device=u.device)
    for t in range(len(k) - 2, -1, -1):
        c = torch.roll(u, lo + t, axis) + k[t]
        less = c < m
        m = torch.where(less, c, m)
        a = torch.where(less, lo + t, a)
    return m, a


def _windows(p):
    return [_window(n, p["dx"][a], p["h"], p["P"][a], p["W"][a]) for a, n in enumerate(p["shape"])]


def _advance(p, u, steps, per_step=False):
    win = _windows(p)
    hV = p["h"] * p["V"]
    for n in range(steps):
        for a, (lo, k) in enumerate(win):
            u = _axis_min(u, a, lo, k)
        u = u - (hV[n] if per_step else hV)
    return u


def _exact_adjoint(case, seed):
    p = _problem(case, seed)
    win, hV = _windows(p), p["h"] * p["V"]
    u, path = p["u0"], []
    for _ in range(case["steps"]):
        step = []
        for a, (lo, k) in enumerate(win):
            u, d = _axis_argmin(u, a, lo, k)
            step.append(d.to(torch.int32))
        u = u - hV
        path.append(step)
    g = _cotangent(p["shape"], seed)
    Pbar, Vbar = torch.zeros(2, dtype=torch.float64, device="cuda"), torch.zeros_like(g)
    for step in reversed(path):
        Vbar -= p["h"] * g
        for a in (1, 0):
            d = step[a].to(torch.int64)
            Pbar[a] += (g * (-d * p["dx"][a])).sum()
            n = p["shape"][a]
            i = torch.arange(n, device="cuda").reshape([n if b == a else 1 for b in range(2)])
            g = torch.zeros_like(g).scatter_add_(a, (i - d) % n, g)
    return {"ubar0": g, "Pbar": Pbar, "Vbar": Vbar, "un": u}


def _exact_integral(case, seed):
    p = _integral_terms(case, seed)
    (lo0, k0), (lo1, k1) = _windows(p)
    x = [torch.arange(n, dtype=torch.float64, device="cuda") / n for n in p["shape"]]
    phase = [(2.0 * math.pi * (float(m[0]) * x[0][:, None] + float(m[1]) * x[1][None, :])) for m in p["modes"]]
    cost = []
    for t0, a0 in enumerate(k0):
        for t1, a1 in enumerate(k1):
            S = torch.zeros(p["shape"], dtype=torch.float64, device="cuda")
            for m, c, al in zip(p["modes"], p["coef"], phase):
                th = 2.0 * math.pi * (float(m[0]) * (lo0 + t0) / p["shape"][0]
                                      + float(m[1]) * (lo1 + t1) / p["shape"][1])
                f = complex(math.sin(th) / th, (1.0 - math.cos(th)) / th) if th else 1.0 + 0.0j
                z = complex(c) * f
                S += z.real * torch.cos(al) - z.imag * torch.sin(al)
            cost.append((lo0 + t0, lo1 + t1, (a0 + a1) - p["h"] * S))
    u = p["u0"]
    for _ in range(case["steps"]):
        m = None
        for d0, d1, c in cost:
            v = torch.roll(u + c, (d0, d1), (0, 1))
            m = v if m is None else torch.minimum(m, v)
        u = m
    return u


def exact(case, seed):
    kind = case["kind"]
    if kind == "decomp":
        return None                       # the method's own approximation at eta > 0, not the scheme's value
    if kind == "integral":
        return _exact_integral(case, seed)
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if kind == "batch":
        us, rows = [], []
        for p in _instances(case, seed):
            u = _advance(p, p["u0"], case["steps"])
            r = (u - p["u0"]) / (case["steps"] * p["h"])
            us.append(u)
            rows.append([-float(r.mean()), -float(r.max()), -float(r.min())])
        return {"u": us, "hbar": np.array(rows)}
    p = _problem(case, seed)
    if kind == "step":
        return {"u": _advance(p, p["u0"], 1), "argmin": None}
    return _advance(p, p["u0"], case["steps"], per_step=(kind == "run_tv"))
