"""Edges of the ring kernels' dispatch rules: the cluster-resident kernel's slice
sizes, and the FitzHugh-Nagumo slope in integer or FP64 arithmetic; the sine's
reduction edges."""
import numpy as np
import pytest

import oracle
from paper_2410_19075_gb300 import inputs as I
from _common import PARAMS, inputs_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("N,R", [(129, 64), (257, 1), (1025, 256), (1921, 960), (4095, 2000), (4096, 2047),
                                 (5120, 700), (8191, 4095), (8192, 1)])
def test_cluster_slices_equal_streaming_bitwise(model, N, R):
    """Slice sizes with a ragged last slice and windows up to the whole ring; the
    slope read after the run comes from the prefix form the cluster kernel leaves."""
    from paper_2410_19075_gb300 import Network
    y0, npar = inputs_for(model, 0, N, 11 + N)
    outs = []
    for streaming in (False, True):
        with Network(model, 0, N, R, PARAMS[model](), streaming=streaming) as net:
            if npar is not None:
                net.set_node_param(npar)
            net.set_state(y0)
            net.step(19, 0.01)
            outs.append((net.get_state(), net.observables(), net.rhs()))
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("R", [1, 31, 32, 63, 64, 1000])  # the integer form needs windows of 65 nodes
@pytest.mark.parametrize("sigma,a", [(0.1, 0.5), (3.5, 0.5), (4.5, 0.5), (100.0, -2.0), (0.1, 63.9), (0.1, 64.0)])
def test_fhn_slope_both_forms_match_oracle(R, sigma, a):
    """sigma and a on both sides of the integer form's range (coupling constants
    below 2^62, |a| < 64).  Both forms and the oracle round each term of the slope's
    bracket to a few 2^-53 of its size; 1e-12 of the largest slope covers the
    oracle's sum of up to 2000 terms."""
    from paper_2410_19075_gb300 import Network
    N = 5000
    params = I.fhn_params(sigma=sigma, a=a)
    y0, _ = inputs_for(1, 0, N, 5 + R)
    q = np.arange(0, N, 7)
    with Network(1, 0, N, R, params) as net:
        net.set_state(y0)
        k = net.rhs().reshape(2, N)[:, q]
    ref = oracle.rhs_sampled(1, 0, N, R, params, y0, q)
    assert np.abs(k - ref).max() < 1e-12 * max(1.0, np.abs(ref).max())


def test_hh_rates_over_the_voltage_range():
    """The gates' slopes over |V| < 256 mV and next to the removable singularities at
    -40 and -55 mV (series below 0.625 mV from them).  alpha - (alpha + beta) x cancels,
    so the bound is 1e-14 of alpha + beta (the rates' error is below 2^-52 and the oracle's
    libm and cancellation a few times that; 1 - exp(-x) at 0.06 loses four bits there)."""
    from paper_2410_19075_gb300 import Network
    rng = np.random.default_rng(9)
    near = np.concatenate([s + d * sgn for s in (-40.0, -55.0) for sgn in (-1, 1)
                           for d in [np.array([0.0, 1e-9, 0.624, 0.625, 0.626, 0.9])]])
    V = np.concatenate([near, np.linspace(-255.9, 255.9, 1999), rng.uniform(-90, 50, 2000)])
    N, R = V.size, 3
    gates = rng.uniform(0.0, 1.0, 3 * N)
    params = I.hh_params()
    y0 = np.concatenate([V, gates])
    for streaming in (False, True):
        with Network(2, 0, N, R, params, streaming=streaming) as net:
            net.set_state(y0)
            k = net.rhs().reshape(4, N)
        ref = oracle.rhs_sampled(2, 0, N, R, params, y0, np.arange(N))
        zero, one = y0.copy(), y0.copy()
        zero[N:], one[N:] = 0.0, 1.0
        alpha = oracle.rhs_sampled(2, 0, N, R, params, zero, np.arange(N))[1:]
        beta = -oracle.rhs_sampled(2, 0, N, R, params, one, np.arange(N))[1:]
        assert (np.abs(k[1:] - ref[1:]) / (alpha + beta)).max() < 1e-14
        assert np.abs(k[0] - ref[0]).max() < 1e-12 * np.abs(ref[0]).max()


@pytest.mark.parametrize("N", [5, 255, 256, 257, 16385, 131072, 131073])
@pytest.mark.parametrize("model", [0, 1])
def test_link_matrix_prefix_forms(model, N):
    """A ring written as rows, on both sides of the size (512 sub-tiles) up to which every
    CTA scans the sub-tile totals itself, against the ring kernels: both add the same exact
    sums, and convert them with roundings of 2^-53 of the slope's terms (1e-12)."""
    from paper_2410_19075_gb300 import Network
    R = 2
    cols = (np.arange(N)[:, None] + np.array([d for d in range(-R, R + 1) if d])) % N
    y0, _ = inputs_for(model, 0, N, 3 + N)
    outs = []
    for rows in (False, True):
        net = (Network.from_links(model, N, np.arange(N + 1) * 2 * R, cols.ravel(), PARAMS[model]()) if rows
               else Network(model, 0, N, R, PARAMS[model](), streaming=True))
        net.set_state(y0)
        k = net.rhs()
        net.step(3, 0.01)
        outs.append((k, net.get_state(), net.observables(), net.dp5(t_end=0.1, rtol=1e-6, atol=1e-6, h0=0.01)["status"],
                     net.get_state()))
        net.close()
    for a, b in zip(*outs):
        assert np.abs(np.asarray(a) - np.asarray(b)).max(initial=0.0) < 1e-12 * max(1.0, np.abs(outs[0][0]).max())


@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_sincos_reduction_edges(sign):
    """sin and cos next to every point where the reduction changes its table entry or
    quadrant.  The routine's error is below 2^-53.6 and its conversion rounds by 2^-54,
    numpy's rounds by 2^-54: 2e-16 in all."""
    from paper_2410_19075_gb300.sim import math_eval
    j = np.concatenate([np.arange(0, 4 * 1024 + 2), np.arange(0, 166800, 1024), [166885, 166886]])
    x = [j * (np.pi / 2048)]
    for d in (np.inf, -np.inf):
        e = x[0]
        for _ in range(3):
            e = np.nextafter(e, d)
            x.append(e)
    x = sign * np.concatenate(x)
    x = x[np.abs(x) < 256]
    s, c = math_eval(0, x), math_eval(1, x)
    assert np.abs(s - np.sin(x)).max() < 2e-16 and np.abs(c - np.cos(x)).max() < 2e-16
    assert np.abs(s).max() <= 1.0 and np.abs(c).max() <= 1.0
