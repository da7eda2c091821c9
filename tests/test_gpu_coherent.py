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


@pytest.mark.parametrize("n_rings,N,R", [(200, 1024, 350), (200, 1023, 350), (200, 1000, 7), (160, 2048, 128), (24, 8192, 700),
                                         (24, 7937, 700)])
@pytest.mark.parametrize("model,phase", [(0, 0.0), (0, np.pi / 2), (3, 0.0)])
def test_batched_dormand_prince_of_rings_in_phase(model, phase, n_rings, N, R):
    """Batches large enough that a CTA takes as many nodes as it can, every node's sine or
    cosine exactly 2^53 on its grid: the streaming kernels' bits."""
    from paper_2410_19075_gb300 import Batch
    y0 = _state(model, N, phase, 0.0)
    opts = dict(t_end=0.3, rtol=1e-7, atol=1e-8, h0=0.1, out_dt=0.1)
    outs = []
    for n, streaming in ((n_rings, False), (1, True)):
        nets = [_net(model, N, R, y0, streaming) for _ in range(n)]
        with Batch(nets) as batch:
            stats = batch.dp5([opts] * n)
        outs.append([(st, net.get_state(), net.observables()) for st, net in zip(stats, nets)])
        for net in nets:
            net.close()
    st, y, order = outs[1][0]
    assert np.abs(order - 1.0).max() < 1e-12
    for got in outs[0]:
        assert got[0] == st and np.array_equal(got[1], y) and np.array_equal(got[2], order)
