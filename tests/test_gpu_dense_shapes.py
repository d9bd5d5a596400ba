"""Shapes where the register-tile searches change over: windows at the bounds of
the flat, scanned and shared-pivot searches, lanes forced so that each takes
lines it would not by itself, ragged last segments, row blocks, both storage
types, smooth fields with shocks, noise and exact ties.  Values, argmins and
window-edge counts against the oracle, bit for bit."""
import numpy as np
import pytest

from edge_counts import edge_hits
from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# shape, W, lanes per line (0: the library's choice), h
CASES = [
    ((5, 191), (2, 47), 0, 0.05),          # 95 displacements: flat
    ((5, 197), (2, 48), 0, 0.05),          # 97: banded where lanes are forced
    ((5, 197), (2, 48), 16, 0.05),
    ((197, 6), (48, 1), 16, 0.05),
    ((4, 640), (1, 150), 64, 0.03),        # 301, 11 rows a lane
    ((3, 1200), (1, 255), 128, 0.02),      # 511: scanned
    ((3, 1200), (1, 257), 128, 0.02),      # 515: pivots shared by a warp
    ((1200, 4), (300, 1), 128, 0.02),
    ((4, 700), (1, 0), 64, 0.05),          # full window, several warps a line
    ((6, 333), (1, 0), 32, 0.05),
    ((9000,), (700,), 256, 2e-4),          # row blocks
    ((2, 2000), (0, 260), 64, 1e-3),
]


def _fields(shape, kind, seed):
    rng = np.random.default_rng([seed, len(shape), shape[-1]])
    g = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    if kind == "noise":
        return 0.05 * rng.normal(size=shape), 0.1 * rng.normal(size=shape)
    if kind == "ties":
        return rng.integers(0, 4, size=shape) / 64.0, rng.integers(0, 4, size=shape) / 64.0
    u = None
    for _ in range(5):
        f = sum(0.2 * rng.normal() * np.cos(2 * np.pi * (rng.integers(1, 4) * x + rng.random())) for x in g)
        u = f if u is None else np.minimum(u, f)
    return u, 0.3 * np.cos(4 * np.pi * g[-1])


@pytest.mark.parametrize("kind", ["shocks", "noise", "ties"])
@pytest.mark.parametrize("f32", [False, True], ids=["f64", "f32"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "%s-%s-%s" % ("x".join(map(str, c[0])), c[1][-1], c[2]))
def test_bitwise(case, f32, kind, monkeypatch):
    from paper_1210_4090_gb300 import hjlo
    shape, W, lanes, h = case
    if lanes:
        monkeypatch.setenv("HJLO_LANES_PER_LINE", str(lanes))
    u0, V = _fields(shape, kind, 5)
    if f32:
        u0 = u0.astype(np.float32)
    dx = tuple(1.0 / n for n in shape)
    P = (0.25,) * len(shape)
    ref, ref_am = O.run(u0, dx, h, P, W, V, 2, record_argmin=True)
    plan = hjlo.Plan(shape, dx, h, P, W, dtype=hjlo.F32_STORAGE if f32 else hjlo.F64, algo=hjlo.ALGO_MONGE)
    u, Vt = torch.tensor(u0, device="cuda"), torch.tensor(V, device="cuda")
    am = torch.empty((2, len(shape)) + shape, dtype=torch.int32, device="cuda")
    for n in range(2):
        plan.step(u, u, Vt, argmin=am[n])
    cnt = plan.sync()
    plan.close()
    view = np.int32 if f32 else np.int64
    assert np.array_equal(u.cpu().numpy().view(view), ref.view(view))
    assert np.array_equal(am.cpu().numpy(), ref_am.reshape(am.shape))
    assert cnt["error_flags"] == 0
    assert cnt["window_edge_hits"] == edge_hits(u0, dx, h, P, W, V, 2)
