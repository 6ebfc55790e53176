"""The density-error statistic to the last bits: with one particle, err_l2 is the
square of err_max, which the device forms by one FP64 division of the same two
FP32 values."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_the_error_of_one_particle_is_squared_in_full(precision):
    from paper_1906_07925_gb300 import Relaxation
    for s0 in np.linspace(0.021, 0.12, 60):
        p = W.uniform_square_2d(8, 1).copy(s0=float(s0))
        r = Relaxation(p, 1, 1, precision=precision)
        r.set_state(np.array([[0.4, 0.6]]), np.zeros(1, np.uint8))
        r.step(1)
        st = r.stats()
        r.close()
        e = st["err_max"]
        assert 0.1 < e < 1.0
        # err_max: the quotient rounded to 2^-53, then one exact subtraction; err_l2: exact terms, a few FP64 roundings
        assert abs(st["err_l2"] - e * e) <= 2 * e * 2.0 ** -53 + 4 * 2.0 ** -53 * e * e
