"""The adjoint's transpose at the edges of its launch shapes: a line whose
shared memory leaves no room for the table of derivatives, many short lines per
CTA, and lines shorter than a CTA's threads per line.  Bit for bit against the
oracle (the sum for P within its rounding order)."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,W,h", [((6500,), 9, 1e-3), ((5, 6200), (1, 7), 1e-3), ((700, 9), (20, 2), 0.05),
                                       ((9, 700), (2, 20), 0.05), ((40, 3, 50), (4, 0, 5), 0.05)], ids=str)
def test_adjoint_lines(shape, W, h):
    from paper_1210_4090_gb300 import hjlo
    rng = np.random.default_rng(len(shape) + shape[0])
    nd, n = len(shape), 3
    dx, P = tuple(1.0 / s for s in shape), (0.3, -0.2, 0.1)[:nd]
    u0, V, ub = rng.normal(size=shape) * 0.05, rng.normal(size=shape) * 0.1, rng.normal(size=shape)
    if nd == 1:
        dx, P = dx[0], P[0]
    plan = hjlo.Plan(shape, dx, h, P, W)
    g0, gP, gV, un = plan.adjoint(torch.tensor(u0, device="cuda"), torch.tensor(V, device="cuda"), n,
                                  torch.tensor(ub, device="cuda"), 2, want_un=True)
    r0, rP, rV = O.adjoint(u0, dx, h, P, W, V, n, ub)
    assert np.array_equal(g0.cpu().numpy().view(np.int64), r0.view(np.int64))
    assert np.array_equal(gV.cpu().numpy().view(np.int64), rV.view(np.int64))
    assert np.array_equal(un.cpu().numpy().view(np.int64), O.run(u0, dx, h, P, W, V, n).view(np.int64))
    # sums of npts products per pass in another order: u = 2^-53 per operation
    scale = np.abs(ub).sum() * n * max(np.max(np.abs(O.table(shape[a], np.atleast_1d(dx)[a], h, np.atleast_1d(P)[a],
                                                             np.atleast_1d(W)[a])[2])) for a in range(nd)) + 1.0
    assert np.max(np.abs(gP.cpu().numpy() - np.atleast_1d(rP))) <= 1e-9 * scale
    plan.close()
