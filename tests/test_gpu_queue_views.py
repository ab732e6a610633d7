"""The dense view of what waits in the queues, its sums and its gathered entries, with
runs of 1 to 64 synapses pending; and a look at them takes no more than some tens of
microseconds on a small network."""
import time

import numpy as np
import pytest

import oracle
from test_gpu_small_rows import _case, _net

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,voxels", [(3001, 30, 1), (20_011, 100, 2), (40_003, 70, 200)])
def test_views_of_queued_runs(n, K, voxels):
    d, csr = _case(n, K, 0, 0)
    rng = np.random.default_rng(n)
    vp, starts = d["vparams"], np.linspace(0, n, voxels + 1).astype(np.int64)
    d.update(n_vox=voxels, voxel_start=starts, vparams=np.tile(vp, (voxels, 1)), d_max=4,
             delay_vv=rng.integers(1, 5, (voxels, voxels)).astype(np.uint8))
    net = _net(d, csr, delivery="queue", event_queue_capacity=400_000)
    ref = oracle.OracleNet(d, "f32")
    for k in (7, 60):
        net.step(k)
        ref.run(k)
        ring = ref.get_state()[3]
        np.testing.assert_array_equal(net.get_state()[3], ring)
        np.testing.assert_array_equal(net.ring_slot_sums(), ring.astype(np.int64).sum(axis=2))
        idx = rng.choice(n, 300, replace=False)
        np.testing.assert_array_equal(net.get_ring_at(idx), ring[:, :, idx].transpose(2, 0, 1))
    assert np.count_nonzero(ring) > 100


def test_a_look_at_the_queues_is_quick():
    """Ten neurons' entries of 20,000: 72 us from queues of events, 222 with the runs
    of one queue after the other read by one thread each; in the ring layout no
    queue is read."""
    d, csr = _case(20_000, 100, 0, 0)
    rng = np.random.default_rng(1)
    d.update(n_vox=2, voxel_start=np.array([0, 10_000, 20_000]), vparams=np.tile(d["vparams"], (2, 1)), d_max=3,
             delay_vv=np.array([[1, 2], [3, 1]], np.uint8))
    idx = rng.choice(20_000, 10, replace=False)
    us = []
    for kw in (dict(delivery="ring"), dict(delivery="queue")):
        net = _net(d, csr, **kw)
        net.step(300)
        t = []
        for _ in range(100):
            t0 = time.perf_counter()
            net.get_ring_at(idx)
            t.append(time.perf_counter() - t0)
        us.append(np.median(t) * 1e6)
    assert us[1] < us[0] + 120, us
