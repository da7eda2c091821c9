"""Hodgkin-Huxley rates at voltages of the 2^-46 grid whose exponentials lie just below a
power of two, where rounding to double carries into the exponent."""
import numpy as np
import pytest

import oracle
from paper_2410_19075_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("streaming", [False, True])
def test_rates_that_round_up_to_a_power_of_two(streaming):
    """exp(-(V + 65)/80) = 4 and exp(-(V + 65)/18) a power of two to within 2^-54. Bound: 1e-14 of
    alpha + beta (rates within 2^-52, and the oracle's libm)."""
    from paper_2410_19075_gb300 import Network
    V = np.array([-175.90354888959126, 109.67308950110622, 246.91623125197538, -202.24314175086917, -65.0])
    assert np.array_equal(np.round(V * 2.0 ** 46), V * 2.0 ** 46)
    N, R = V.size, 1
    params = I.hh_params()
    for gate in (0.0, 0.5, 1.0):
        y0 = np.concatenate([V, np.full(3 * N, gate)])
        with Network(2, 0, N, R, params, streaming=streaming) as net:
            net.set_state(y0)
            k = net.rhs().reshape(4, N)[1:]
        ref = oracle.rhs_sampled(2, 0, N, R, params, y0, np.arange(N))[1:]
        zero, one = (np.concatenate([V, np.full(3 * N, g)]) for g in (0.0, 1.0))
        scale = oracle.rhs_sampled(2, 0, N, R, params, zero, np.arange(N))[1:] - \
            oracle.rhs_sampled(2, 0, N, R, params, one, np.arange(N))[1:]
        assert (np.abs(k - ref) / scale).max() < 1e-14
