"""Lone lines with windows of up to 96 displacements on the GPU, at lengths where the
row blocks change their size or their search: values and argmins are brute force's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("f32", [False, True], ids=["f64", "f32"])
@pytest.mark.parametrize("W", [7, 9, 47])
@pytest.mark.parametrize("N", [4863, 4864, 9727, 9728, 77823, 77824, 77825, 155649, 262145, 525312, 525465])
def test_as_brute_force(N, W, f32):
    from paper_1210_4090_gb300 import hjlo
    rng = np.random.default_rng([N, W])
    x = np.arange(N) / N
    u = 0.3 * np.cos(2 * np.pi * x) + 10.0 ** rng.uniform(-6, 0) * rng.normal(size=N)
    t = torch.tensor(u.astype(np.float32 if f32 else np.float64), device="cuda")
    got = []
    for algo in (hjlo.ALGO_MONGE, hjlo.ALGO_BRUTE):
        plan = hjlo.Plan((N,), 1.0 / N, W / N, 0.2, W, dtype=hjlo.F32_STORAGE if f32 else hjlo.F64, algo=algo)
        out, am = torch.empty_like(t), torch.empty((1, N), dtype=torch.int32, device="cuda")
        plan.step(t, out, None, argmin=am)
        assert plan.sync()["error_flags"] == 0
        plan.close()
        got.append((out.view(torch.int32 if f32 else torch.int64), am))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
