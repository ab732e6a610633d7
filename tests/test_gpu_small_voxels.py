"""A small network of as many voxels as neurons: a call of one step takes no longer
than with the general kernels (a queue capacity of the caller's asks for them), and
both give the same."""
import time

import numpy as np
import pytest

from helpers import custom_net, params_row

pytestmark = pytest.mark.gpu


def test_one_step_calls_on_3000_voxels():
    from paper_2308_01241_gb300 import dtb

    n, K = 3000, 100
    rng = np.random.default_rng(1)
    starts = np.arange(n + 1)
    pre, cls = rng.integers(0, n, (n, K)), rng.random((n, K)) < 0.2
    w = rng.integers(1600, 6400, (n, K)).astype(np.int32)
    d = custom_net(n, pre, cls, w, params_row(), voxel_start=starts, delay_vv=rng.integers(1, 4, (n, n)).astype(np.uint8),
                   d_max=3, nu_ext=2000.0, w_ext=int(2.4 * 65536))
    order = np.argsort(pre.ravel(), kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(pre.ravel(), minlength=n))
    word = (np.repeat(np.arange(n, dtype=np.int64), K)[order] | (cls.ravel()[order].astype(np.int64) << 30))
    out, us = [], []
    for kw in (dict(delivery="ring"), dict(delivery="queue", event_queue_capacity=100_000)):
        net = dtb.Network(n=n, voxel_start=starts, vparams=d["vparams"], delay_vv=d["delay_vv"], d_max=3,
                          csr=(row_ptr, word.astype(np.uint32), w.ravel()[order]), wfmt="int32", wshift=0, dt=d["dt"],
                          nu_ext=d["nu_ext"], w_ext=d["w_ext"], seed=d["seed"], init_seed=d["init_seed"],
                          bold=d["bold"], **kw)
        net.step(300)
        t = []
        for _ in range(40):
            t0 = time.perf_counter()
            net.step(1)
            t.append(time.perf_counter() - t0)
        us.append(np.median(t) * 1e6)
        out.append(net.get_state() + (net.voxel_spikes(),))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    assert out[0][-1].sum() > 1000
    assert us[0] < 0.9 * us[1], us
