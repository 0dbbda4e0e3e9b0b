"""sw_launch_count counts the kernels that each call launches."""
import numpy as np
import pytest

from _helpers import gpu, turbulence

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_counts_per_call(prec):
    lm = gpu()
    N = 32
    uvh = np.ascontiguousarray(np.stack(turbulence(N)))
    h = lm.sw_create(lm.make_params(N, 5e-3, precision=prec, nu8=1e-9), uvh)
    try:
        def launched(call):
            n = lm.sw_launch_count(h)
            r = call()
            return lm.sw_launch_count(h) - n, r
        # a column and a row pass per four fields
        assert launched(lambda: lm.sw_get_fields(h, np.zeros((3, N, N))))[0] == 2
        assert launched(lambda: lm.sw_set_fields(h, uvh))[0] == 2
        # u, v, h, zeta in one pair of passes, then two reductions
        assert launched(lambda: lm.sw_diag(h))[0] == 4
        assert launched(lambda: lm.sw_spectrum(h, np.ascontiguousarray(uvh[0]), N))[0] == 3
        # layout conversion of all fields and their compensation terms
        n, blob = launched(lambda: lm.sw_get_state(h))
        assert n == 1
        assert launched(lambda: lm.sw_set_state(h, blob))[0] == 1
        # the transforms before the first stage, then row and column kernel per stage
        assert launched(lambda: lm.sw_step(h, 3))[0] == 1 + 3 * 4 * 2
    finally:
        lm.sw_destroy(h)
