"""The surrogate MLP at the edges of its kernels' tiles: batches around 32 and
64 rows and the 64-row chunks, one and many input and output columns, one to
seven hidden layers, and widths that take the general kernels.  Predictions,
every gradient and one Adam step against the FP64 oracle, within the FP32
tolerances of mlp_bounds.py."""
import numpy as np
import pytest

from mlp_bounds import assert_within, backward_sigma, forward_sigma, output_grad_sigma, setup
from oracle import mlp as ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_in,width,depth,n_out", [
    (1, 1, 256, 1, 1), (31, 12, 256, 3, 6), (33, 17, 256, 2, 16), (64, 64, 256, 3, 8), (65, 65, 256, 1, 9),
    (4901, 12, 256, 3, 6), (300, 256, 256, 7, 3), (130, 12, 64, 2, 6), (130, 300, 256, 2, 6), (130, 12, 256, 2, 17)])
def test_sizes_match_oracle(B, n_in, width, depth, n_out):
    import torch

    from paper_2308_01241_gb300.surrogate_mlp import MLP

    params, x, t = setup(B=B, n_in=n_in, width=width, depth=depth, n_out=n_out, seed=B)
    net = MLP(params, n_in, width, depth, n_out, max_batch=B)
    dx, dt_ = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = torch.zeros((B, n_out), dtype=torch.float32, device="cuda")
    net.forward(dx, y)
    p16 = [(ref.bf16(W), np.float32(b).astype(np.float64)) for W, b in params]
    yr, cache = ref.forward(p16, ref.bf16(x), bf16_acts=True)
    sa, sz, sy = forward_sigma(p16, cache, yr)
    assert_within(y.cpu().numpy(), yr, sy, "forward output")
    grads, loss = net.gradients(dx, dt_)
    want, dy = ref.loss_and_grad_out(yr, t)
    assert abs(loss - want) < 1e-2 * want
    gr = ref.backward(p16, cache, dy, bf16_acts=True)
    sig = backward_sigma(p16, cache, sa, sz, output_grad_sigma(sy, dy), ref.bf16(dy))
    for li, ((gw, gb), (rw, rb), (sw, sb)) in enumerate(zip(grads, gr, sig)):
        assert_within(gw, rw, sw, f"dW[{li}]")
        assert_within(gb, rb, sb, f"db[{li}]")
    # one Adam step applies exactly these gradients
    assert abs(net.train_step(dx, dt_, lr=1e-3) - loss) <= 1e-6 * loss
    p = [(np.float32(W).astype(np.float64), np.float32(b).astype(np.float64)) for W, b in params]
    ref.adam(p, [(gw.astype(np.float64), gb.astype(np.float64)) for gw, gb in grads], ref.adam_state(p), lr=1e-3)
    for (gw, gb), (rw, rb) in zip(net.params(), p):
        np.testing.assert_allclose(gw, rw, rtol=1e-5, atol=1e-6)
        np.testing.assert_allclose(gb, rb, rtol=1e-5, atol=1e-6)
    net.close()
