"""Hodgkin-Huxley gates: rates at voltages of the 2^-46 grid whose exponentials lie just below a
power of two, where rounding to double carries into the exponent; slopes over the gates' range."""
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


@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (0.95, 1.0), (1.0 - 1e-6, 1.0), (0.0, 1e-6)])
def test_gate_slopes_keep_their_relative_accuracy(lo, hi):
    """alpha (1 - x) - beta x within 2^-50 of alpha (1 - x) + beta x: each rate within 2^-52 and its
    rounding, 1 - x, the products and the difference 2^-53 each.  x / (1 - exp(-x)) cancels next to its
    series (four bits), so voltages within 8 mV of -40 and -55 are left out.  Reference: long double."""
    from paper_2410_19075_gb300 import Network
    rng = np.random.default_rng(12)
    V = np.round(rng.uniform(-100.0, 60.0, 30000) * 2.0 ** 40) / 2.0 ** 40
    V = V[(np.abs(V + 40) > 8) & (np.abs(V + 55) > 8)]
    N = V.size
    x = rng.uniform(lo, hi, (3, N))
    with Network(2, 0, N, 3, I.hh_params(), streaming=True) as net:
        net.set_state(np.concatenate([V, x.ravel()]))
        k = net.rhs().reshape(4, N)[1:]
    v, xl = V.astype(np.longdouble), x.astype(np.longdouble)
    over = [z / -np.expm1(-z) for z in ((v + 40) / 10, (v + 55) / 10)]
    alpha = np.stack([over[0], 7 * np.exp(-(v + 65) / 20) / 100, over[1] / 10])
    beta = np.stack([4 * np.exp(-(v + 65) / 18), 1 / (1 + np.exp(-(v + 35) / 10)), np.exp(-(v + 65) / 80) / 8])
    gain, loss = alpha * (1 - xl), beta * xl
    assert (np.abs(k - (gain - loss)) / (gain + loss)).max() < 2.0 ** -50
