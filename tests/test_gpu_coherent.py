"""Coherent states of small Kuramoto rings inside one thread-block cluster: the sums
of sine and cosine over the ring reach N 2^53, past 64 bits from 1024 nodes on."""
import numpy as np
import pytest

from _common import PARAMS

pytestmark = pytest.mark.gpu

SIZES = [(1000, 350), (1025, 1), (4000, 10), (4096, 127), (5000, 250), (8192, 400)]


def _state(model, N, phase, spread):
    phi = phase + spread * np.random.default_rng(N).uniform(-1.0, 1.0, N)
    return phi if model == 0 else np.concatenate([phi, 0.01 * np.ones(N)])


def _net(model, N, R, y0, streaming):
    from paper_2410_19075_gb300 import Network
    net = Network(model, 0, N, R, PARAMS[model](), streaming=streaming)
    net.set_state(y0)
    return net


def _run(model, N, R, y0, streaming, dp5):
    """RK4 steps or a Dormand-Prince run, the slope, and a batched step from the prefix it leaves."""
    from paper_2410_19075_gb300 import Batch
    with _net(model, N, R, y0, streaming) as net:
        if dp5:
            st = net.dp5(t_end=0.5, rtol=1e-7, atol=1e-8, h0=0.1, out_dt=0.1)
            assert st["status"] == 0
        else:
            net.step(5, 0.01)
        out = [net.get_state(), net.rhs()]
        with Batch([net]) as batch:
            batch.step(2, 0.01)
            batch.sync()
        return out + [net.get_state(), net.observables()]


@pytest.mark.parametrize("dp5", [False, True])
@pytest.mark.parametrize("model", [0, 3])
@pytest.mark.parametrize("phase,spread", [(0.3, 0.0), (3.0, 0.0), (-1.5, 1e-3), (0.0, 1.5)])
@pytest.mark.parametrize("N,R", SIZES)
def test_order_parameter_of_coherent_rings(N, R, phase, spread, model, dp5):
    """Every recorded R, the state and the slope, bit for bit the streaming kernels', and the
    loaded state's R against numpy: a sum of N terms with an error of at most N 2^-53 each (1e-12)."""
    y0 = _state(model, N, phase, spread)
    outs = [_run(model, N, R, y0, streaming, dp5) for streaming in (False, True)]
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
    R0 = abs(np.exp(1j * y0[:N]).mean())
    order = outs[0][3]
    assert order.size > 3 and abs(order[0] - R0) < 1e-12
    assert abs(order[1] - R0) < 1e-2  # 0.01 time units on (Dormand-Prince: the run's own R(t0))
    if spread == 0.0:  # identical nodes stay identical
        assert np.abs(order - 1.0).max() < 1e-12
