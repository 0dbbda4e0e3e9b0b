"""Cell index and weight of displacements by integer arithmetic (floor_int) against
floor, through the lift: next to integers, over its range and beyond it."""
import numpy as np
import pytest

from _helpers import gpu
from oracle.remap import grid, lift

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CELLS = [0, 1, 2, 3, 7, 2 ** 15, 2 ** 23, 2 ** 29, 2 ** 30 - 1, 2 ** 30, 2 ** 30 + 1, 2 ** 31 - 1, 2 ** 31, 2 ** 33 + 5, 2 ** 40,
         2 ** 51 + 1, 2 ** 53]
FRACTIONS = [0.0, 0.5, 0.25, 1.0 - 2.0 ** -20, 2.0 ** -22, 2.0 ** -30, 2.0 ** -52, 1e-300]


@pytest.mark.parametrize("N", [16, 256])
def test_lift_at_edges_of_cells_bitwise(N):
    lm = gpu()
    rng = np.random.default_rng(N)
    X, Y = grid(N)
    dx = 2.0 * np.pi / N

    def positions(base):
        d = rng.choice(CELLS, base.shape).astype(np.float64) + rng.choice(FRACTIONS, base.shape)
        d *= rng.choice([-1.0, 1.0], base.shape) * dx
        for _ in range(3):  # up to three units to either side
            d = np.where(rng.random(base.shape) < 0.5, np.nextafter(d, rng.choice([-np.inf, np.inf], base.shape)), d)
        return base + d

    px, py = positions(X), positions(Y)
    f = {"a": rng.standard_normal((N, N)), "b": np.cos(2 * X + Y)}
    dev = {k: torch.from_numpy(v).cuda() for k, v in f.items()}
    g = lm.lmean_lift(torch.from_numpy(px).cuda(), torch.from_numpy(py).cuda(), dev)
    ref = lift(f, px, py)
    for k in f:
        assert np.array_equal(g[k].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_lift_non_finite(bad):
    lm = gpu()
    N = 16
    X, Y = grid(N)
    px = X.copy()
    px[3, 5] = bad
    f = torch.from_numpy(np.cos(2 * X + Y)).cuda()
    g = lm.lmean_lift(torch.from_numpy(px).cuda(), torch.from_numpy(Y.copy()).cuda(), {"a": f})["a"].cpu().numpy()
    ok = np.ones((N, N), bool)
    ok[3, 5] = False
    assert np.isnan(g[3, 5]) and np.array_equal(g[ok], f.cpu().numpy()[ok])
