"""The column stage's launch variants (blocks in quarters, halves and whole) give
the same bits for every model, stepper and scheme, and the whole blocks of large
grids match the oracle under another stepper than RK4."""
import numpy as np
import pytest

from _helpers import gpu, turbulence
from oracle import SWOracle, rel_l2

pytestmark = pytest.mark.gpu

RUNS = {
    "euler2d": (dict(model="euler2d"), dict(strategy=1, fields=("zeta", "u"))),
    "euler2d-heun-s2": (dict(model="euler2d", stepper="heun"), dict(strategy=2, fields=("zeta", "v"))),
    "kinematic": (dict(model="kinematic", adv=(0.3, -0.2)), dict(strategy=1, fields=("h", "q"))),
    "kinematic-euler-s2": (dict(model="kinematic", adv=(0.3, -0.2), stepper="euler"), dict(strategy=2, fields=("h", "q"))),
    "heun": (dict(stepper="heun", visc="laplace"), dict(strategy=1, fields=("zeta", "q"))),
    "euler": (dict(stepper="euler"), dict(strategy=1, fields=("zeta", "h"))),
    "xi-first": (dict(stepper="euler"), dict(strategy=2, fields=("u", "q"), scheme="xi_first")),
    "rk4-q": (dict(), dict(strategy=1, fields=("h", "q"))),
}


def _open(lm, N, prec, par, lmp, n, seed):
    h = lm.sw_create(lm.make_params(N, 5e-3, precision=prec, nu8=1e-9, **par),
                     np.ascontiguousarray(np.stack(turbulence(N, seed=seed))))
    lm.lmean_begin(h, lm.make_lm_params(n_steps=n, **lmp))
    return h


def _close(lm, h, N, lmp):
    out = {k: np.zeros((N, N)) for k in lmp["fields"] + ("pos_x", "pos_y") + tuple("e_" + f for f in lmp["fields"])}
    lm.lmean_end(h, out)
    out["uvh"] = np.zeros((3, N, N))
    lm.sw_get_fields(h, out["uvh"])
    lm.sw_destroy(h)
    return out


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("name", sorted(RUNS))
def test_quarters_halves_and_whole_blocks_bitwise(name, prec):
    """Alone at 64^2, among 8 runs and among 14: two means and positions take 48
    column blocks a run, so these are 48 (quarters), 384 (halves) and 672 (whole)."""
    lm = gpu()
    par, lmp = RUNS[name]
    N, n, ref = 64, 4, None
    for members in (1, 8, 14):
        hs = [_open(lm, N, prec, par, lmp, n, 1001 + i) for i in range(members)]
        b = lm.sw_batch_create(hs)
        lm.sw_batch_step(b, n)
        lm.sw_batch_destroy(b)
        outs = [_close(lm, h, N, lmp) for h in hs]
        ref = ref or outs[0]
        for k in ref:
            assert np.isfinite(ref[k]).all() and np.array_equal(ref[k], outs[0][k]), (members, k)


@pytest.mark.parametrize("stepper", ["heun", "euler"])
def test_large_grid_other_steppers(stepper):
    """FP64 at 1024^2 (256-thread whole blocks, one mode at a time) against the oracle."""
    lm = gpu()
    N, n = 1024, 2
    uvh = turbulence(N)
    lmp = dict(strategy=1, fields=("zeta", "q"))
    h = lm.sw_create(lm.make_params(N, 5e-3, stepper=stepper, nu8=10.0 / 341.0 ** 8), np.ascontiguousarray(np.stack(uvh)))
    lm.lmean_begin(h, lm.make_lm_params(n_steps=n, pos=False, **lmp))
    lm.lmean_step(h, n)
    out = {k: np.zeros((N, N)) for k in ("zeta", "q", "e_zeta", "e_q")}
    lm.lmean_end(h, out)
    lm.sw_destroy(h)
    o = SWOracle(N, 5e-3, *uvh, stepper=stepper, nu8=10.0 / 341.0 ** 8)
    o.lmean_begin(1, fields=("zeta", "q"), pos=False, eulerian=True, n_steps=n)
    o.lmean_step(n)
    r = o.lmean_end()
    for k in ("zeta", "q"):
        assert rel_l2(out[k], r[k]) < 1e-12 and rel_l2(out["e_" + k], r["E_" + k]) < 1e-12, k
