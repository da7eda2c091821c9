"""Kuramoto rings with inertia on both sides of the sizes whose sub-tiles are resident at once
only with more CTAs per SM (another compilation of the same kernel): against one node per thread."""
import numpy as np
import pytest

from _common import PARAMS, inputs_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edge", [7, 8])
@pytest.mark.parametrize("offset", [-1, 0, 1])
def test_ring_sizes_around_one_wave(edge, offset, tmp_path):
    import torch
    from paper_2410_19075_gb300 import Network
    from paper_2410_19075_gb300.sim import tune_clear, tune_load
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 256 * (edge * sms + offset) - 3
    R = N // 3
    y0, _ = inputs_for(3, 0, N, 9)
    outs = []
    for npt in (2, 1):
        f = tmp_path / f"tune{npt}"
        f.write_text(f"# kind model a b npt flat\n0 3 {N} {R} {npt} 1\n")
        tune_clear()
        tune_load(str(f))
        try:
            with Network(3, 0, N, R, PARAMS[3]()) as net:
                assert net.tune_info()["npt"] == npt
                net.set_state(y0)
                net.step(3, 0.01)
                outs.append((net.get_state(), net.observables(), net.rhs()))
        finally:
            tune_clear()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
