"""Dormand-Prince runs of link matrices: the kernels between them."""
import numpy as np
import pytest

from _common import PARAMS, inputs_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [600, 131072, 131073])  # both prefix forms of the RK4 kernels (512 sub-tiles)
def test_no_memset_between_the_launches_of_an_attempt(model, N):
    """A run's graph of attempts holds kernels only (a memset node costs more than a stage's gather), and
    RK4 steps after the run go on from its state as after loading that state."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    from paper_2410_19075_gb300 import Network
    cols = (np.arange(N)[:, None] + np.array([-2, -1, 1, 2])) % N
    y0, npar = inputs_for(model, 0, N, N)
    with Network.from_links(model, N, np.arange(N + 1) * 4, cols.ravel(), PARAMS[model]()) as net:
        if npar is not None:
            net.set_node_param(npar)
        net.set_state(y0)
        opts = dict(t_end=0.2, rtol=1e-7, atol=1e-8, h0=0.01)
        net.dp5(**opts)
        net.set_state(y0)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]):  # the first one of a process sees nothing
            torch.zeros(1, device="cuda")
            torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            st = net.dp5(**opts)
        events = [e.name for e in prof.events()]
        y = net.get_state()
        net.step(3, 0.01)
        after = net.get_state(), net.rhs()
        net.set_state(y)
        net.step(3, 0.01)
        for a, b in zip(after, (net.get_state(), net.rhs())):
            assert np.array_equal(a, b)
    assert st["status"] == 0
    attempts = st["accepted"] + st["rejected"]
    kernels = sum("graph_stage_kernel" in e for e in events)
    memsets = sum(e.startswith("Memset") for e in events)  # on the device
    if kernels == 0:
        pytest.skip("the profiler saw no kernels")
    assert kernels >= 6 * attempts
    assert memsets <= 2  # the prologues at the run's start and end
