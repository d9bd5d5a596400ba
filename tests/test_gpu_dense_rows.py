"""The register-tile searches on the GPU at rows whose nearest rival differs by
less than the screen's error (the lines of test_dense_rows.py): every value and
argmin is the definition's, on whole lines and in row blocks, each search.  (Line lengths
that are no powers of two: the tables of those fall on the screen's units.)"""
import numpy as np
import pytest

from test_dense_rows import _rivals, _table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(u, W, h, monkeypatch, env):
    """One pass along the last axis of u (lines, points): values, argmins, block rows and segment."""
    from paper_1210_4090_gb300 import hjlo
    for name, v in env.items():
        monkeypatch.setenv(name, str(v))
    # along the other axis a unit step costs 1e3^2 / 2h: its pass leaves u as it is
    plan = hjlo.Plan(u.shape, (1e3, 1.0 / u.shape[1]), h, (0.0, 0.0), (1, W), algo=hjlo.ALGO_MONGE)
    out = torch.empty(u.shape, dtype=torch.float64, device="cuda")
    am = torch.empty((2,) + u.shape, dtype=torch.int32, device="cuda")
    plan.step(torch.tensor(u, device="cuda"), out, None, argmin=am)
    cnt, info = plan.sync(), plan.info()
    plan.close()
    assert cnt["error_flags"] == 0 and int(am[0].abs().max()) == 0
    return out.cpu().numpy(), am[1].cpu().numpy(), info


def _expect(u, k, W):
    """The definition on the periodic lines u."""
    val, am = np.empty_like(u), np.empty(u.shape, np.int32)
    w = len(k)
    for i in range(len(u)):
        lifted = np.concatenate([u[i][-W:], u[i], u[i][:W]])
        c = np.lib.stride_tricks.sliding_window_view(lifted, w) + k
        t = c.argmin(1)
        val[i], am[i] = c[np.arange(len(t)), t], W - t
    return val, am


# points, W, lanes a line, the search they make (hjlo_dense.cuh): flat, 9, 13 or 11 rows a segment
@pytest.mark.parametrize("ends", [True, False], ids=["ends", "anywhere"])
@pytest.mark.parametrize("N,W,lanes", [(250, 40, 16), (280, 60, 32), (410, 60, 32), (1200, 257, 128)],
                         ids=["flat", "9", "13", "11"])
def test_whole_lines(N, W, lanes, ends, monkeypatch):
    rng = np.random.default_rng([N, ends])
    h, k = 0.02, _table(2 * W + 1, 1.0 / N, 0.02)
    u = np.empty((1500 if N < 1000 else 400, N))
    for i in range(len(u)):
        u[i] = np.roll(_rivals(rng, N, k, N, ends), -W)       # halo index j is point j - W
    got, am, _ = _run(u, W, h, monkeypatch, {"HJLO_LANES_PER_LINE": lanes})
    val, ram = _expect(u, k, W)
    assert np.array_equal(got.view(np.int64), val.view(np.int64))
    assert np.array_equal(am, ram)


@pytest.mark.parametrize("N,W,rows", [(4100, 40, 300), (4100, 100, 400), (4100, 100, 700), (9100, 400, 900)],
                         ids=["flat", "9", "13", "11"])
def test_first_rows_of_row_blocks(N, W, rows, monkeypatch):
    rng = np.random.default_rng([N, W, rows])
    h, w, k = 0.02, 2 * W + 1, _table(2 * W + 1, 1.0 / N, 0.02)
    u = np.empty((70, N))
    for i in range(len(u)):
        parts = [_rivals(rng, rows + w - 1, k, rows, True)[:w + 8] for _ in range(N // rows)]
        u[i] = max(q.max() for q in parts)
        for b, q in enumerate(parts):
            u[i, (b * rows - W + np.arange(w + 8)) % N] = q
    got, am, info = _run(u, W, h, monkeypatch, {"HJLO_BLOCK_ROWS": rows})
    assert info["row_blocks"][1] > 1 and info["block_rows"][1] == rows
    val, ram = _expect(u, k, W)
    assert np.array_equal(got.view(np.int64), val.view(np.int64))
    assert np.array_equal(am, ram)
