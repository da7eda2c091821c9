"""Dormand-Prince runs of batches that mix models, sizes and topologies, whose groups of
small rings run beside one another and beside the captured graphs of the other members."""
import numpy as np
import pytest

from _common import PARAMS, inputs_for

pytestmark = pytest.mark.gpu

# (model, topology, N, R, attempts of at most this length): rings of every cluster size, rings
# larger than a cluster, a cube, a ball, a link matrix
MEMBERS = [(m, 0, n, max(1, int(0.3 * n)), 0.2) for m in range(4) for n in (65, 400, 700, 1500, 3000, 8000)] + \
    [(0, 0, 9000, 2000, 0.2), (1, 0, 12000, 3000, 0.2), (0, 1, 12, 2, 0.2), (3, 2, 11, 3, 0.2), (0, 4, 600, 3, 0.2)] + \
    [(0, 0, 500, 100, 0.0015), (3, 0, 900, 300, 0.004), (0, 0, 10000, 100, 0.02)]


def _net(model, topo, N, R):
    from paper_2410_19075_gb300 import Network
    if topo == 4:
        cols = (np.arange(N)[:, None] + np.array([d for d in range(-R, R + 1) if d])) % N
        net = Network.from_links(model, N, np.arange(N + 1) * 2 * R, cols.ravel(), PARAMS[model]())
        topo = 0
    else:
        net = Network(model, topo, N, R, PARAMS[model]())
    y0, npar = inputs_for(model, topo, N, 70 + N)
    if npar is not None:
        net.set_node_param(npar)
    net.set_state(y0)
    return net


@pytest.mark.parametrize("members", [MEMBERS, MEMBERS[:24], MEMBERS[18:24] + MEMBERS[29:31], MEMBERS[24:]])
def test_members_equal_runs_alone(members):
    """Members with small step limits take up to 1000 attempts, four launches of their group."""
    from paper_2410_19075_gb300 import Batch
    opts = [dict(t_end=1.5, rtol=1e-7, atol=1e-8, h0=0.2, h_max=h, out_dt=0.11) for *_, h in members]
    nets = [_net(*m[:4]) for m in members]
    with Batch(nets) as batch:
        for _ in range(2):  # the second run on the streams of the first
            stats = batch.dp5(opts)
    got = [(st, net.get_state(), net.observables(), net.rhs()) for st, net in zip(stats, nets)]
    for m, o, g, net in zip(members, opts, got, nets):
        net.close()
        with _net(*m[:4]) as alone:
            alone.dp5(**o)
            st = alone.dp5(**o)
            assert g[0] == st and st["status"] == 0
            for a, b in zip(g[1:], (alone.get_state(), alone.observables(), alone.rhs())):
                assert np.array_equal(a, b)
