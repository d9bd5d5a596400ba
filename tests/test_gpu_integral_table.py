"""The first discrete semigroup with the plan's table of path costs and without
it (HJLO_TEST_COST_BYTES=0 sums them in the step) give the same bits: the same
binary64 operations on the same operands, in 1D-3D, with ragged sizes, full
windows, more outputs than a block holds, infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((1,), 0, 1), ((33,), 5, 3), ((31,), 0, 2), ((13, 37), (2, 3), 5), ((32, 32), (4, 4), 2), ((5, 6, 7), (1, 2, 0), 3)]


@pytest.mark.parametrize("special", [False, True], ids=["finite", "inf-nan"])
@pytest.mark.parametrize("shape,W,nmodes", CASES, ids=lambda v: str(v))
def test_table_and_sum_agree(shape, W, nmodes, special, monkeypatch):
    from paper_1210_4090_gb300 import hjlo
    rng = np.random.default_rng([7, len(shape), nmodes])
    modes = rng.integers(-3, 4, size=(nmodes, len(shape)))
    coef = rng.normal(size=nmodes) + 1j * rng.normal(size=nmodes)
    u0 = rng.normal(size=shape)
    if special:
        u0.reshape(-1)[0] = np.nan
        u0.reshape(-1)[-1] = -np.inf
        u0.reshape(-1)[u0.size // 2] = np.inf
    out = []
    for limit in (None, "0"):
        if limit is not None:
            monkeypatch.setenv("HJLO_TEST_COST_BYTES", limit)
        plan = hjlo.IntegralPlan(shape, tuple(1.0 / n for n in shape), 0.05, (0.3,) * len(shape), W, modes, coef)
        u = torch.tensor(u0, device="cuda")
        plan.run(u, 3)
        plan.sync()
        plan.close()
        out.append(u.cpu().numpy())
    assert np.array_equal(out[0].view(np.int64), out[1].view(np.int64))
