"""Tiles that the register-tile searches leave to divide and conquer: one line
of a tile far from the others or with an infinity, and fields too large for the
table's curvature.  Every value and argmin is the definition's, and only the
lines that fail the rounding margin themselves go to brute force."""
import numpy as np
import pytest

from test_dense_rows import _table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

H = 0.02


def _pass(u, k, W):
    """The definition along the last axis in binary64: values, argmins."""
    u = np.asarray(u, np.float64)
    lifted = np.concatenate([u[:, u.shape[1] - W:], u, u[:, :W]], axis=1)
    c = np.lib.stride_tricks.sliding_window_view(lifted, len(k), axis=1) + k
    t = c.argmin(2)
    return np.take_along_axis(c, t[..., None], 2)[..., 0], (W - t).astype(np.int32)


def _failing(u, k):
    """Lines (last axis) that fail the rounding margin."""
    a = np.abs(np.asarray(u, np.float64)).max(1) + np.abs(k).max()
    return int((~(np.diff(k, 2).min() > a * 2.0 ** -49)).sum())


# points, W, lanes a line, rows a block: flat, 9, 13, 11 rows a segment, and 9 in row blocks
@pytest.mark.parametrize("f32", [False, True], ids=["f64", "f32"])
@pytest.mark.parametrize("strided", [False, True], ids=["contig", "strided"])
@pytest.mark.parametrize("N,W,lanes,rows", [(250, 40, 16, 0), (280, 60, 32, 0), (410, 60, 32, 0), (1200, 257, 128, 0),
                                            (4100, 100, 0, 400)], ids=["flat", "9", "13", "11", "blocks"])
@pytest.mark.parametrize("kind", ["one far", "one infinite", "large"])
def test_left_tiles(kind, N, W, lanes, rows, strided, f32, monkeypatch):
    from paper_1210_4090_gb300 import hjlo
    if rows and strided:
        pytest.skip("row blocks are for contiguous axes")
    if lanes:
        monkeypatch.setenv("HJLO_LANES_PER_LINE", str(lanes))
    if rows:
        monkeypatch.setenv("HJLO_BLOCK_ROWS", str(rows))
    L = 70
    rng = np.random.default_rng([N, len(kind)])
    x = np.arange(N) / N
    u = np.stack([np.minimum(0.3 * np.cos(2 * np.pi * (x + rng.random())), 0.2 * np.cos(4 * np.pi * (x + rng.random())))
                  + 0.01 * rng.normal(size=N) for _ in range(L)])
    if kind == "one far":
        u[37] += 1e12
    elif kind == "one infinite":
        u[37, N // 3] = np.inf
    else:
        u *= 1e6
    u = u.astype(np.float32 if f32 else np.float64)
    k, k1 = _table(2 * W + 1, 1.0 / N, H), _table(3, 1e6, H)      # the other axis: a step costs 2.5e13
    trunc = (lambda v: v.astype(np.float32)) if f32 else (lambda v: v)
    if strided:
        val, am = _pass(u, k, W)
        val = trunc(val)
        fail = _failing(u, k) + _failing(val.T, k1)
        ref = trunc(_pass(val.T, k1, 1)[0]).T
    else:
        mid = trunc(_pass(u.T, k1, 1)[0]).T
        fail = _failing(u.T, k1)
        ref, am = _pass(mid, k, W)
        ref = trunc(ref)
        if rows:                                                  # a block's lines by themselves: the span it stages
            for b in range(-(-N // rows)):
                at = (b * rows - W + np.arange(rows + 2 * W)) % N
                fail += _failing(mid[:, at], k)
        else:
            fail += _failing(mid, k)
    shape, dx, ax = ((N, L), (1.0 / N, 1e6), 0) if strided else ((L, N), (1e6, 1.0 / N), 1)
    plan = hjlo.Plan(shape, dx, H, (0.0, 0.0), (W, 1) if strided else (1, W), algo=hjlo.ALGO_MONGE,
                     dtype=hjlo.F32_STORAGE if f32 else hjlo.F64)
    assert (plan.info()["row_blocks"][1] > 1) == bool(rows)
    inp = torch.tensor(np.ascontiguousarray(u.T if strided else u), device="cuda")
    out = torch.empty_like(inp)
    args = torch.empty((2,) + shape, dtype=torch.int32, device="cuda")
    plan.step(inp, out, None, argmin=args)
    cnt = plan.sync()
    plan.close()
    got, gam = out.cpu().numpy(), args[ax].cpu().numpy()
    view = np.int32 if f32 else np.int64
    want = np.ascontiguousarray(ref.T if strided else ref)
    assert np.array_equal(got.view(view), want.view(view))
    assert np.array_equal(gam.T if strided else gam, am)
    assert cnt["error_flags"] == 0 and cnt["brute_fallback_lines"] == fail
    assert kind == "large" or 0 < fail < L
