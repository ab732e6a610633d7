"""The bins layout on small networks, which by default keep the queue layout: a
bin capacity of the caller's asks for real bins.  Rasters and the whole state
(delay ring included) against the C oracle for every weight format, both
channel modes, the OU drive, voxels wider than the delivery window, both
schedules and a checkpoint; and the default layout of the same network gives
the same."""
import numpy as np
import pytest

import oracle
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu
OU = dict(mu=0.1, sigma=0.15, tau=5.0)


def _case(wfmt, n_ch, wide):
    if wide:  # one voxel of 300,000 neurons, delay 1
        tb = ng.make_tables(dict(ng.load_config("c1_single_voxel_1k"), wfmt=wfmt), n_neurons=300_000, K=40)
    else:
        tb = ng.make_tables(dict(ng.load_config("c2_multi_voxel_1m"), gain={"default": 1.35}), n_neurons=60013, n_vox=9,
                            K=80)
    pre, cls, wbin = ng.host_pull(tb)
    rng = np.random.default_rng(3)
    if n_ch == 4:
        cls = rng.integers(0, 4, size=cls.shape).astype(np.uint8)
    pull = (pre, cls, wbin)
    d = ng.oracle_inputs(tb, pull, wfmt="int16" if wfmt == "int8" else wfmt)
    d["n_ch"] = n_ch
    if wfmt == "int8":  # with a power-of-two scale per source
        q = ((wbin.astype(np.int32) % 120) + 1).astype(np.int8)
        rs = rng.integers(0, 4, size=tb.n).astype(np.uint8)
        d.update(wfmt=oracle.W_INT8, w=q, wshift=8, pre_shift=rs)
        row_ptr, word, wb = ng.host_push(tb, (pre, cls, q.view(np.uint8).astype(np.uint16)))
        csr = (row_ptr, word, wb.astype(np.uint8).view(np.int8), rs)
    else:
        row_ptr, word, wb = ng.host_push(tb, pull)
        csr = (row_ptr, word, tb.wtable(wfmt)[wb])
    return tb, d, csr


@pytest.mark.parametrize("wfmt,n_ch,ou,wide", [("int16", 2, False, False), ("int32", 2, False, False),
                                               ("bf16", 2, True, False), ("int8", 2, False, False),
                                               ("int16", 4, False, False), ("int32", 4, True, False),
                                               ("int16", 2, False, True)])
def test_small_bins_match_the_oracle(wfmt, n_ch, ou, wide):
    from paper_2308_01241_gb300 import dtb

    tb, d, csr = _case(wfmt, n_ch, wide)
    if ou:
        d["ou"] = OU
    ref = oracle.OracleNet(d, "f32")
    nets = [dtb.Network(n=tb.n, voxel_start=tb.voxel_start, vparams=d["vparams"], delay_vv=tb.delay_vv, d_max=tb.d_max,
                        csr=csr, wfmt=wfmt, wshift=d["wshift"], n_ch=n_ch, dt=d["dt"], nu_ext=d["nu_ext"],
                        w_ext=d["w_ext"], seed=d["seed"], init_seed=d["init_seed"], bold=d["bold"], delivery="bins",
                        bin_capacity=cap, ou=OU if ou else None) for cap in (20000, 0)]
    total = 0
    for k, sched in ((1, -1), (40, 0), (70, 1)):
        rids, roff = ref.run(k)
        total += len(rids)
        for net in nets:
            net.set_schedule(sched)
            net.step(k)
            ids, off = net.get_spikes()
            np.testing.assert_array_equal(off, roff)
            np.testing.assert_array_equal(ids, rids)
    assert total > 500
    want = ref.get_state()
    for net in nets:
        for a, b in zip(net.get_state(), want):
            np.testing.assert_array_equal(a, b)
        assert net.counters()[0] == ref.events()
    np.testing.assert_array_equal(nets[0].ring_slot_sums(), nets[1].ring_slot_sums())
    # each layout's checkpoint resumes in the other
    blobs = [net.save_state() for net in nets]
    assert blobs[0] == blobs[1]
    rids, _ = ref.run(30)
    for net, blob in zip(nets, reversed(blobs)):
        net.load_state(blob)
        net.step(30)
        np.testing.assert_array_equal(net.get_spikes()[0], rids)
