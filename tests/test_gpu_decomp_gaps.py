"""The whole-period decomposition's emission where points with many vertices
and long stretches without any (the inside of concave components) alternate in
a write-back block: rough stretches at the line's ends, across its seam and
between blocks, one rough line among smooth ones.  Several CTAs share the rows
of a block that many components reach; blocks of few rows, of rows that do not
divide, and more blocks than are shared (rows 1).  Bit for bit the oracle's method, with its number of components."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(shape, W, u0, eta):
    from paper_1210_4090_gb300 import hjlo as H
    nd = len(shape)
    dx, h, P = tuple(1.0 / s for s in shape), 0.02, (0.3,) * nd
    plan = H.Plan(shape, dx, h, P, (W,) * nd, algo=H.ALGO_DECOMP)
    plan.set_tolerance(eta)
    assert all(c > 0 for c in plan.info()["split_chunks"][:nd])
    u = torch.tensor(u0, device="cuda")
    plan.run(u, None, 2)
    cnt = plan.sync()
    plan.close()
    ref, ncomp = O.decomp_run(u0, dx, h, P, (W,) * nd, None, 2, eta)
    assert np.array_equal(u.cpu().numpy().view(np.int64), np.asarray(ref).view(np.int64))
    assert cnt["components"] == ncomp and cnt["error_flags"] == 0


@pytest.mark.parametrize("rows", ["1", "3", "40", "257", "2000"])
@pytest.mark.parametrize("at", [0, 700, 1950])
def test_rough_stretch(at, rows, monkeypatch):
    monkeypatch.setenv("HJLO_DECOMP_SPLIT", "1")
    monkeypatch.setenv("HJLO_DECOMP_CHUNK", "96")
    monkeypatch.setenv("HJLO_DECOMP_SPLIT_ROWS", rows)
    N = 2000
    u0 = 0.1 * np.sin(2 * np.pi * np.arange(N) / N)
    q = (at + np.arange(120)) % N
    u0[q] += 0.01 * np.random.default_rng(at + 5).normal(size=120)
    _check((N,), 60, u0, 1e-6)


@pytest.mark.parametrize("rough", [0, 4, 8])
def test_rough_line_among_smooth(rough, monkeypatch):
    monkeypatch.setenv("HJLO_DECOMP_SPLIT", "1")
    monkeypatch.setenv("HJLO_DECOMP_SPLIT_ROWS", "90")
    shape = (9, 500)
    u0 = np.tile(0.1 * np.sin(2 * np.pi * np.arange(500) / 500), (9, 1))
    u0[rough, 200:330] += 0.01 * np.random.default_rng(rough).normal(size=130)
    _check(shape, 4, u0, 1e-6)
