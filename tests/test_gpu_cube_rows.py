"""Cubes on both sides of the row length from which the node pass asks for a share of the L1:
stepped alone and in a batch (whose launches never ask), the same bits."""
import pytest

from _common import PARAMS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,N1", [(0, 360), (0, 361), (3, 448), (3, 449)])
def test_node_pass_row_lengths(model, N1):
    import torch
    from paper_2410_19075_gb300 import Batch, Network
    n = N1 ** 3 * (2 if model == 3 else 1)
    y0 = torch.rand(n, device="cuda", dtype=torch.float64, generator=torch.Generator("cuda").manual_seed(N1))
    outs = []
    for batched in (False, True):
        with Network(model, 1, N1, 3, PARAMS[model]()) as net:
            net.set_state(y0)
            if batched:
                with Batch([net]) as b:
                    b.step(2, 0.01)
                    b.sync()
            else:
                net.step(2, 0.01)
            out = torch.empty_like(y0)
            net.get_state_device(out)
            outs.append((out, net.observables()))
    assert torch.equal(outs[0][0], outs[1][0])
    assert (outs[0][1] == outs[1][1]).all() and outs[0][1].size == 3
