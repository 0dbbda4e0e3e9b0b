"""The stage kernels' launch variants give the same bits: blocks split in two
halves (small launches) and whole ones, products split over blocks and not,
one replay and several; and kinematic dynamics of any grid sizes in a batch."""
import numpy as np
import pytest

from _helpers import FIELDS, gpu, turbulence
from oracle import SWOracle, rel_l2

pytestmark = pytest.mark.gpu


def _open(lm, N, prec, strategy, n, seed=1001):
    K = (N - 1) // 3
    h = lm.sw_create(lm.make_params(N, 5e-3, precision=prec, nu8=10.0 / K ** 8),
                     np.ascontiguousarray(np.stack(turbulence(N, seed=seed))))
    lm.lmean_begin(h, lm.make_lm_params(strategy, FIELDS + ("q",), n_steps=n))
    return h


def _close(lm, h, N):
    out = {k: np.zeros((N, N)) for k in FIELDS + ("q", "pos_x", "pos_y", "e_zeta", "e_q")}
    lm.lmean_end(h, out)
    lm.sw_destroy(h)
    return out


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("N,strategy", [(64, 1), (64, 2), (256, 1), (256, 2)])
def test_large_batch_matches_alone_bitwise(N, strategy, prec):
    """A run alone (split column blocks; at 64^2 one product per row block)
    against the same run among enough others that blocks are whole."""
    lm = gpu()
    n = 3
    h = _open(lm, N, prec, strategy, n)
    lm.lmean_step(h, n)
    ref = _close(lm, h, N)
    hs = [_open(lm, N, prec, strategy, n, seed=1001 + i) for i in range(96 if N == 64 else 12)]
    b = lm.sw_batch_create(hs)
    lm.sw_batch_step(b, n)
    lm.sw_batch_destroy(b)
    outs = [_close(lm, h, N) for h in hs]
    for k in ref:
        assert np.array_equal(ref[k], outs[0][k]), k


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("strategy", [1, 2])
def test_replays_split_bitwise(strategy, prec):
    """Eleven steps in one call (graphs of 8 and 1 steps and the final step)
    and one by one (a transform-only start each)."""
    lm = gpu()
    res = []
    for chunks in ([11], [1] * 11, [8, 3]):
        h = _open(lm, 64, prec, strategy, 11)
        for c in chunks:
            lm.lmean_step(h, c)
        res.append(_close(lm, h, 64))
    for r in res[1:]:
        for k in r:
            assert np.array_equal(res[0][k], r[k]), k


@pytest.mark.parametrize("stepper", ["rk4", "heun", "euler"])
def test_kinematic_batch_of_any_sizes(stepper):
    """Kinematic dynamics has no transforms: grids of any sizes share a batch."""
    lm = gpu()
    sizes, hs, os_ = (16, 64, 1024), [], []
    for N in sizes:
        u, v, h = turbulence(N)
        kw = dict(model="kinematic", adv=(0.3, -0.2), nu8=1e-9 if N < 100 else 0.0)
        hs.append(lm.sw_create(lm.make_params(N, 5e-3, stepper=stepper, **kw),
                               np.ascontiguousarray(np.stack([u, v, h]))))
        os_.append(SWOracle(N, 5e-3, u, v, h, stepper=stepper, **kw))
    b = lm.sw_batch_create(hs)
    lm.sw_batch_step(b, 2)
    lm.sw_batch_destroy(b)
    for N, h, o in zip(sizes, hs, os_):
        out = np.zeros((3, N, N))
        lm.sw_get_fields(h, out)
        lm.sw_destroy(h)
        o.step(2)
        ref = np.stack(o.fields())
        assert rel_l2(out[0], ref[0]) < 1e-12 and rel_l2(out[1], ref[1]) < 1e-12, N
