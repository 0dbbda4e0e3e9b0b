"""Kinematic dynamics (no averages, so no transforms): a pointwise kernel of its
own, alone and beside runs with transforms."""
import numpy as np
import pytest

from _helpers import gpu, turbulence
from oracle import SWOracle, rel_l2

pytestmark = pytest.mark.gpu
ADV = (0.3, -0.2)


def _create(lm, N, prec="f64", stepper="rk4", visc="hyper8", **kw):
    kw = kw or dict(model="kinematic", adv=ADV)
    return lm.sw_create(lm.make_params(N, 5e-3, precision=prec, stepper=stepper, visc=visc, nu8=1e-9, **kw),
                        np.ascontiguousarray(np.stack(turbulence(N))))


def _fields(lm, h, N):
    out = np.zeros((3, N, N))
    lm.sw_get_fields(h, out)
    lm.sw_destroy(h)
    return out


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("N", [16, 512, 2048])
def test_own_kernel(N, prec):
    """One launch per stage, of the pointwise kernel: the column stage's blocks
    (255 registers in FP64, exchange buffers allocated) took twice its time."""
    lm = gpu()
    h = _create(lm, N, prec)
    kt = lm.sw_kernel_times(h, 2)
    lm.sw_destroy(h)
    assert {k: c for k, (_, c, _) in kt.items() if c} == {"update": 8}


@pytest.mark.parametrize("visc", ["hyper8", "laplace"])
@pytest.mark.parametrize("stepper", ["rk4", "heun", "euler"])
@pytest.mark.parametrize("N", [16, 512, 1024])
def test_against_oracle(N, stepper, visc):
    """All three fields, the depth included (as h - 1)."""
    lm = gpu()
    h = _create(lm, N, stepper=stepper, visc=visc)
    lm.sw_step(h, 3)
    out = _fields(lm, h, N)
    o = SWOracle(N, 5e-3, *turbulence(N), model="kinematic", adv=ADV, stepper=stepper, visc=visc, nu8=1e-9)
    o.step(3)
    ref = np.stack(o.fields())
    out[2] -= 1.0
    ref[2] -= 1.0
    for f in range(3):
        assert rel_l2(out[f], ref[f]) < 1e-12, f


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("stepper", ["rk4", "heun", "euler"])
def test_beside_transforms_bitwise(stepper, prec):
    lm = gpu()
    alone = []
    for members in range(2):
        runs = [(2048, {}), (64, {}), (128, dict(f0=1.0)), (16, {})]
        hs = [_create(lm, N, prec, stepper, **kw) for N, kw in runs]
        if members == 0:
            for h in hs:
                lm.sw_step(h, 9)
        else:
            b = lm.sw_batch_create(hs)
            lm.sw_batch_step(b, 9)
            lm.sw_batch_destroy(b)
        res = [_fields(lm, h, N) for h, (N, _) in zip(hs, runs)]
        if members == 0:
            alone = res
    for a, r in zip(alone, res):
        assert np.array_equal(a, r)
