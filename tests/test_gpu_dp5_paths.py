"""Dormand-Prince runs of small rings inside one cluster against the seven launches per
attempt of larger rings (SIM_FLAG_STREAMING selects those): the same bits, alone and
in batches that give a ring another number of CTAs."""
import numpy as np
import pytest

from _common import PARAMS, inputs_for

pytestmark = pytest.mark.gpu

OPTS = dict(t_end=1.5, rtol=1e-7, atol=1e-8, h0=0.2, out_dt=0.11)


def _net(model, N, R, streaming=False):
    from paper_2410_19075_gb300 import Network
    net = Network(model, 0, N, R, PARAMS[model](), streaming=streaming)
    y0, npar = inputs_for(model, 0, N, 40 + N)
    if npar is not None:
        net.set_node_param(npar)
    net.set_state(y0)
    return net


def _outcome(net, st):
    out = [st, net.get_state(), net.observables(), net.rhs()]
    net.step(3, 0.01)
    return out + [net.get_state()]


def _same(a, b):
    assert a[0] == b[0]
    for x, y in zip(a[1:], b[1:]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("N,R", [(3, 1), (33, 16), (257, 128), (1000, 350), (1025, 7), (2049, 700), (4096, 2047), (8192, 100),
                                 (8193, 100)])
def test_cluster_run_equals_streaming_run(model, N, R):
    outs = []
    for streaming in (False, True):
        with _net(model, N, R, streaming) as net:
            outs.append(_outcome(net, net.dp5(**OPTS)))
    _same(*outs)
    assert outs[0][0]["status"] == 0


@pytest.mark.parametrize("model", [0, 1, 2, 3])
def test_batch_members_equal_runs_alone(model):
    from paper_2410_19075_gb300 import Batch
    sizes = [(100 + 61 * i, 1 + 17 * i) for i in range(40)] + [(3000, 1200), (9000, 3000)]
    opts = [dict(OPTS, h0=0.05 + 0.01 * (i % 7), rtol=10.0 ** -(6 + i % 3)) for i in range(len(sizes))]
    nets = [_net(model, N, R) for N, R in sizes]
    batch = Batch(nets)
    got = [_outcome(net, st) for net, st in zip(nets, batch.dp5(opts))]
    batch.close()
    for (N, R), o, g, net in zip(sizes, opts, got, nets):
        net.close()
        with _net(model, N, R) as alone:
            _same(g, _outcome(alone, alone.dp5(**o)))


def test_attempts_over_several_launches_and_budget():
    """More attempts than one launch makes (256), and a budget that ends inside one."""
    for budget in (10 ** 6, 300, 256, 5):
        outs = []
        for streaming in (False, True):
            with _net(0, 500, 100, streaming) as net:
                outs.append(_outcome(net, net.dp5(t_end=3.0, rtol=1e-6, atol=1e-6, h0=0.01, h_max=0.005,
                                                  max_attempts=budget)))
        _same(*outs)
        n = outs[0][0]["accepted"]  # 600 steps of 0.005, and one more if their sum rounds below 3
        assert n in (600, 601) if budget > 601 else n == budget
        assert outs[0][0]["status"] == (0 if budget > 600 else -7)
