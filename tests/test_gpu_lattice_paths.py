"""Edges of the ball's and disk's gather: blocks of one, two and four nodes per
thread (lattice edges 48 and 72 for balls, 400 for disks), ragged blocks, windows as
wide as the lattice, more reads than one table chunk, window arrays and row prefixes.
Edges of the cube's tiles, alone and in a batch."""
import numpy as np
import pytest

import oracle
from paper_2410_19075_gb300 import inputs as I
from _common import nodes_of

pytestmark = pytest.mark.gpu

BALL, DISK = 2, 3


@pytest.mark.parametrize("topo,N,P", [(BALL, 47, 5), (BALL, 48, 1), (BALL, 49, 24), (BALL, 71, 6), (BALL, 72, 4), (BALL, 73, 7),
                                      (BALL, 75, 37), (DISK, 399, 199), (DISK, 400, 7), (DISK, 401, 200), (DISK, 403, 1),
                                      (DISK, 7200, 3500)])
@pytest.mark.parametrize("model", [0, 3])
def test_gather_blocks(topo, N, P, model):
    """Slopes at sampled nodes (every corner of a block and of the lattice among them)
    against the oracle; one step against RK4 of the slopes (both are the same FP64
    expressions up to the stage inputs' rounding, 1e-14); the low-memory form gives the
    same bits."""
    from paper_2410_19075_gb300 import Network
    if N > 7000 and model == 3:
        pytest.skip("one model is enough for the longest rows")
    n = nodes_of(topo, N)
    params = I.ks_params(alpha=1.3) if model == 0 else I.ksi_params(mu=1.0)
    rng = np.random.default_rng(N + P)
    y0 = np.concatenate([rng.uniform(-3.1, 3.1, n)] + ([rng.uniform(-0.1, 0.1, n)] if model == 3 else []))
    edge = [0, 1, N - 2, N - 1]
    corners = [(z * N + j) * N + i for z in (edge if topo == BALL else [0]) for j in edge for i in edge]
    q = np.unique(np.concatenate([corners, rng.choice(n, 40, replace=False)]))
    if P > 300:
        q = q[:: max(1, q.size // 6)]
    outs = []
    for low in (False, True):
        with Network(model, topo, N, P, params, low_memory=low) as net:
            net.set_state(y0)
            k1 = net.rhs()
            net.step(1, 0.01)
            outs.append((k1, net.get_state(), net.observables()))
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
    k1, y1, order = outs[0]
    ref = oracle.rhs_sampled(model, topo, N, P, params, y0, q)
    assert np.abs(k1.reshape(-1, n)[:, q] - ref).max() < 1e-13
    assert abs(order[0] - oracle.order_parameter(y0[:n])) < 1e-12
    with Network(model, topo, N, P, params) as net:
        k, y = [k1], None
        for c in (0.005, 0.005, 0.01):
            net.set_state(y0 + c * k[-1])
            k.append(net.rhs())
    y = y0 + 0.01 / 6.0 * (k[0] + 2.0 * k[1] + 2.0 * k[2] + k[3])
    assert np.abs(y1 - y).max() < 1e-14


@pytest.mark.parametrize("model", [0, 3])
def test_cube_tiles(model):
    """Cubes around the edges of their tiles (16 columns up to edge 297, 8 above), windows
    from the smallest to the whole edge: slopes at sampled nodes against the oracle, and
    all of them in one batch, small and large tiles in the same launches, against the
    same steps alone, bit for bit."""
    from paper_2410_19075_gb300 import Batch, Network
    params = I.ks_params(alpha=1.3) if model == 0 else I.ksi_params(mu=1.0)
    cubes = [(3, 1), (16, 7), (17, 8), (31, 15), (33, 2), (113, 1), (297, 2), (298, 3), (305, 1)]
    rng = np.random.default_rng(5 + model)
    ys, alone, nets = [], [], []
    for N, P in cubes:
        n = N ** 3
        y0 = np.concatenate([rng.uniform(-3.1, 3.1, n)] + ([rng.uniform(-0.1, 0.1, n)] if model == 3 else []))
        ys.append(y0)
        with Network(model, 1, N, P, params) as net:
            net.set_state(y0)
            k1 = net.rhs()
            net.step(2, 0.01)
            alone.append((net.get_state(), net.observables()))
        edge = [0, 1, N - 2, N - 1]
        q = np.unique([(z * N + j) * N + i for z in edge for j in edge for i in edge])
        # window sums: exact but for the rounding onto 2^-F, 1e-13 as for the other lattices
        assert np.abs(k1.reshape(-1, n)[:, q] - oracle.rhs_sampled(model, 1, N, P, params, y0, q)).max() < 1e-13
    try:
        for (N, P), y0 in zip(cubes, ys):
            nets.append(Network(model, 1, N, P, params))
            nets[-1].set_state(y0)
        with Batch(nets) as batch:
            batch.step(2, 0.01)
            batch.sync()
        for net, (y, order) in zip(nets, alone):
            assert np.array_equal(net.get_state(), y)
            assert np.array_equal(net.observables(), order)
    finally:
        for net in nets:
            net.close()
