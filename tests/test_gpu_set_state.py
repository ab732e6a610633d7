"""dtb_set_state with the ring left unchanged and another step: what had spilled
out of a full queue or bin still arrives, at the next step of its ring slot."""
import numpy as np
import pytest

import oracle
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delivery,qcap,bcap", [("queue", 1024, 0), ("bins", 1024, 20000)])
@pytest.mark.parametrize("move,far", [(8, False), (-2, False), (8, True)])
def test_spilled_events_follow_a_moved_step(delivery, qcap, bcap, move, far):
    from paper_2308_01241_gb300 import dtb

    tb = ng.make_tables(dict(ng.load_config("c2_multi_voxel_1m"), gain={"default": 1.45}), n_neurons=200003, n_vox=24,
                        K=100)
    pull = ng.host_pull(tb)
    net = dtb.from_tables(tb, dtb.host_csr(tb, pull), delivery=delivery, event_queue_capacity=qcap, bin_capacity=bcap)
    ref = oracle.OracleNet(ng.oracle_inputs(tb, pull), "f32")
    D = tb.d_max + 1
    net.step(200)
    ref.run(200)
    V, j, r, ring, t = ref.get_state()
    assert np.count_nonzero(ring) > 0
    # a multiple of 2 D keeps every slot, queue, accumulator and bin where it is
    moved = t + move * 2 * D
    assert moved >= 0
    ref.set_state(V, j, r, ring, moved)
    if far:  # by way of the last step there is
        net.set_state(t=2 ** 63 - 1)
    net.set_state(t=moved)
    for k in (1, 2 * D, 40):
        net.step(k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
