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
        # layout conversion of all fields and their compensation terms
        n, blob = launched(lambda: lm.sw_get_state(h))
        assert n == 1
        assert launched(lambda: lm.sw_set_state(h, blob))[0] == 1
    finally:
        lm.sw_destroy(h)
