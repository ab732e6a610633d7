"""More voxels than neurons: voxels may be empty, and there may be 65,535 of them.
At most 3,072 keep the one-CTA steps of small networks, more take the general
kernels; rasters, state and voxel counts against the C oracle around that line."""
import numpy as np
import pytest

import oracle
from helpers import custom_net, params_row

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [3072, 3073, 4000])
@pytest.mark.parametrize("delivery", ["ring", "queue", "bins"])
def test_more_voxels_than_neurons(nv, delivery):
    from paper_2308_01241_gb300 import dtb

    n, K = 301, 12
    rng = np.random.default_rng(nv)
    starts = np.sort(np.append(rng.integers(0, n + 1, nv - 1), [0, n])).astype(np.int64)
    assert (np.diff(starts) == 0).sum() > nv - n - 1
    vp = params_row(g=(0.003, 0.00002, 0.01, 0.0005))
    pre, cls = rng.integers(0, n, (n, K)), rng.integers(0, 2, (n, K))
    w = rng.integers(2000, 40000, (n, K)).astype(np.int32)
    d = custom_net(n, pre, cls, w, vp, voxel_start=starts, delay_vv=rng.integers(1, 4, (nv, nv)).astype(np.uint8),
                   d_max=3, nu_ext=2000.0, w_ext=2 * 65536)
    order = np.argsort(pre.ravel(), kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(pre.ravel(), minlength=n))
    word = (np.repeat(np.arange(n, dtype=np.int64), K)[order] | (cls.ravel()[order] << 30)).astype(np.uint32)
    net = dtb.Network(n=n, voxel_start=starts, vparams=d["vparams"], delay_vv=d["delay_vv"], d_max=3,
                      csr=(row_ptr, word, w.ravel()[order]), wfmt="int32", wshift=0, dt=d["dt"], nu_ext=d["nu_ext"],
                      w_ext=d["w_ext"], seed=d["seed"], init_seed=d["init_seed"], bold=d["bold"], delivery=delivery)
    ref = oracle.OracleNet(d, "f32")
    total = np.zeros(nv, np.int64)
    for k in (1, 40, 150):
        net.step(k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
        total += np.bincount(np.searchsorted(starts, ids, side="right") - 1, minlength=nv)
    assert total.sum() > 100
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(net.voxel_spikes(), total)
