"""The autotuner times a launch shape once: the register-tile searches have no
wide-bracket offload to turn on or off."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# at most 9 shapes an axis (lanes a line and lines a tile halved, kept, doubled), and for row blocks 3 times
# that (rows halved, kept, doubled)
@pytest.mark.parametrize("shape,W,most", [((64, 64, 64), 6, 27), ((20000,), 30, 27)], ids=["grid", "line"])
def test_register_tile_shapes_are_timed_once(shape, W, most):
    from paper_1210_4090_gb300 import hjlo
    nd = len(shape)
    u = torch.tensor(0.1 * np.random.default_rng(4).normal(size=shape), device="cuda")
    plan = hjlo.Plan(shape, tuple(1.0 / n for n in shape), 0.02 if nd > 1 else W / shape[0], (0.0,) * nd, (W,) * nd,
                     algo=hjlo.ALGO_MONGE)
    rep = plan.autotune(u, None, 1)
    plan.close()
    assert 1 <= rep["trials"] <= most
