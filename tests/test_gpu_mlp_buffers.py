"""The surrogate MLP's buffers: a prediction written over its own input gives what
one into a buffer of its own gives, and a batch size whose buffers do not fit the
256-wide path takes the general one."""
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


def test_a_batch_size_that_only_the_general_path_has_room_for():
    """Seven hidden layers, batches of up to 2^17 rows: the 256-wide path keeps seven
    gradients of a batch, the general one two.  With memory left for the latter only,
    the network is created and gives the same, bit for bit."""
    import torch

    from paper_2308_01241_gb300 import dtb
    from paper_2308_01241_gb300.surrogate_mlp import MLP

    B, depth, most = 300, 7, 1 << 17
    params, x, t = setup(B=B, n_in=12, width=256, depth=depth, n_out=6, seed=4)
    dx, dt_ = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()

    def results(net):
        y = torch.zeros((B, 6), device="cuda")
        net.forward(dx, y)
        grads, loss = net.gradients(dx, dt_)
        net.train_step(dx, dt_, 1e-3)
        return [y.cpu().numpy()] + [a for pair in grads + net.params() for a in pair], loss

    net = MLP(params, 12, 256, depth, 6, max_batch=B)
    want, loss = results(net)
    net.close()
    torch.cuda.synchronize()
    row = depth * (2 + 4) * 256 + 2 * 12 + 4 * 6 + 2 * 6  # activations, pre-activations, input, output and its gradient
    general, fused = most * (row + 2 * 512), most * (row + depth * 512)
    assert fused - general > 300 << 20
    free = torch.cuda.mem_get_info()[0]
    ballast = torch.empty(free - (general + fused) // 2, dtype=torch.uint8, device="cuda")
    try:
        net = MLP(params, 12, 256, depth, 6, max_batch=most)
        got, loss2 = results(net)
        net.close()
        with pytest.raises(dtb.DtbError) as e:
            MLP(params, 12, 256, depth, 6, max_batch=2 * most)
        assert e.value.code == dtb.DTB_ENOMEM
    finally:
        del ballast
        torch.cuda.empty_cache()
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
    assert abs(loss2 - loss) <= 1e-6 * loss
