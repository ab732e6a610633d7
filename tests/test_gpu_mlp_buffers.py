"""The surrogate MLP's buffers: a prediction written over its own input gives what
one into a buffer of its own gives."""
import numpy as np
import pytest

from mlp_bounds import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_in,n_out", [(65_536, 12, 6), (40_001, 6, 16), (5_978, 12, 12)])
@pytest.mark.parametrize("where", ["start", "end"])
def test_prediction_over_its_own_input(B, n_in, n_out, where):
    import torch

    from paper_2308_01241_gb300.surrogate_mlp import MLP

    params, x, _ = setup(B=B, n_in=n_in, width=256, depth=3, n_out=n_out, seed=B)
    net = MLP(params, n_in, 256, 3, n_out, max_batch=B)
    want = torch.zeros((B, n_out), device="cuda")
    net.forward(torch.from_numpy(x).cuda(), want)
    room = torch.zeros(B * max(n_in, n_out), device="cuda")
    dx = room[:B * n_in] if n_in >= n_out or where == "start" else room[-B * n_in:]
    dx = dx.view(B, n_in)
    dx.copy_(torch.from_numpy(x))
    y = (room[:B * n_out] if where == "start" else room[-B * n_out:]).view(B, n_out)
    net.forward(dx, y)
    np.testing.assert_array_equal(y.cpu().numpy(), want.cpu().numpy())
    net.close()
