"""Row passes of small grids by teams of groups (one product per block) against
whole chunks of products per block: the same bits, for every kind of product."""
import numpy as np
import pytest

from _helpers import gpu, turbulence

pytestmark = pytest.mark.gpu

ALL = ("zeta", "h", "u", "v", "q")
RUNS = {
    "s1": (dict(), dict(strategy=1, fields=ALL)),
    "s2": (dict(), dict(strategy=2, fields=ALL)),
    "s2-one": (dict(), dict(strategy=2, fields=("u",), eulerian=False)),
    "dynamics": (dict(), None),
    "s1-heun": (dict(stepper="heun", visc="laplace"), dict(strategy=1, fields=("zeta", "q"), pos=False)),
    "s2-xi-first": (dict(stepper="euler"), dict(strategy=2, fields=ALL, scheme="xi_first")),
    "s1-euler2d": (dict(model="euler2d", stepper="heun"), dict(strategy=1, fields=("zeta", "u"))),
    "s2-euler2d": (dict(model="euler2d"), dict(strategy=2, fields=("zeta", "v"))),
    "s1-kinematic": (dict(model="kinematic", adv=(0.3, -0.2)), dict(strategy=1, fields=ALL)),
    "s2-kinematic": (dict(model="kinematic", adv=(0.3, -0.2)), dict(strategy=2, fields=ALL)),
    "positions": (dict(), dict(strategy=2, fields=(), eulerian=False)),
}


def _run(lm, N, prec, par, lmp, choice):
    n = 4
    h = lm.sw_create(lm.make_params(N, 5e-3, precision=prec, nu8=1e-9, **par),
                     np.ascontiguousarray(np.stack(turbulence(N))))
    b = None
    try:
        if lmp:
            lm.lmean_begin(h, lm.make_lm_params(n_steps=n, **lmp))
        if choice is None:
            (lm.lmean_step if lmp else lm.sw_step)(h, n)
        else:
            b = lm.sw_batch_create([h])
            lm.sw_batch_set_shape(b, choice)
            lm.sw_batch_step(b, n)
        out = {}
        if lmp:
            keys = list(lmp["fields"])
            if lmp["strategy"] == 2 or lmp.get("pos", True):
                keys += ["pos_x", "pos_y"]
            if lmp.get("eulerian", True):
                keys += ["e_" + f for f in lmp["fields"]]
            out = {k: np.zeros((N, N)) for k in keys}
            lm.lmean_end(h, out)
        out["uvh"] = np.zeros((3, N, N))
        lm.sw_get_fields(h, out["uvh"])
        return out
    finally:
        if b is not None:
            lm.sw_batch_destroy(b)
        lm.sw_destroy(h)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("N", [16, 32, 64, 128])
@pytest.mark.parametrize("name", sorted(RUNS))
def test_teams_match_whole_chunks_bitwise(name, N, prec):
    """256 points per block, one product (a team) and all of them; also one
    product with the most points (blocks too large for a team from 64^2 on)."""
    lm = gpu()
    par, lmp = RUNS[name]
    ref = _run(lm, N, prec, par, lmp, None)
    for choice in (3, 0, 12):
        got = _run(lm, N, prec, par, lmp, choice)
        for k in ref:
            assert np.isfinite(ref[k]).all() and np.array_equal(ref[k], got[k]), (choice, k)
