"""The bins and queue layouts where requests without capacities get another one.

A bins request without a bin capacity keeps the queue layout up to 28 MiB of
accumulators, and networks of at most 3,072 neurons run in one CTA, so tests that
only name a delivery mode do not reach every layout.  Here the same checks run
with capacities given, which keeps the layout that is named (shown by the counter
hook, whose range starts at that layout's capacity)."""
import numpy as np
import pytest

import oracle
import test_gpu_c2_golden as golden
import test_gpu_edge as edge
import test_gpu_parity as parity
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu

BIN_CAPACITY, QUEUE_CAPACITY = 40_000, 200_000


@pytest.fixture
def dtb(monkeypatch):
    """The binding, with capacities for bins and queue requests that give none."""
    from paper_2308_01241_gb300 import dtb as m

    class Kept(m.Network):
        def __init__(self, *, delivery="ring", bin_capacity=0, event_queue_capacity=0, **kw):
            if delivery == "bins":
                bin_capacity = bin_capacity or BIN_CAPACITY
            elif delivery == "queue":
                event_queue_capacity = event_queue_capacity or QUEUE_CAPACITY
            super().__init__(delivery=delivery, bin_capacity=bin_capacity, event_queue_capacity=event_queue_capacity,
                             **kw)

    monkeypatch.setattr(m, "Network", Kept)
    return m


def test_capacities_keep_the_layout(dtb):
    """Counters below a capacity are refused: a bin holds 40,000 events, one of a
    step's eight queues 25,000 runs (both rounded up to whole lines), and the ring
    has none."""
    tb = ng.make_tables(ng.load_config("c1_single_voxel_1k"))
    csr = dtb.host_csr(tb, ng.host_pull(tb))
    for delivery, kw, low, code in (("bins", dict(event_queue_capacity=5000), 39_999, dtb.DTB_EINVAL),
                                    ("queue", {}, 24_999, dtb.DTB_EINVAL), ("ring", {}, 1 << 32, dtb.DTB_ESTATE)):
        net = dtb.from_tables(tb, csr, delivery=delivery, **kw)
        with pytest.raises(dtb.DtbError) as e:
            net.test_preset_counters(low)
        assert e.value.code == code
        if delivery != "ring":
            net.test_preset_counters(low + 200)


@pytest.mark.parametrize("delivery", ["bins", "queue", "ring"])
@pytest.mark.parametrize("wfmt", ["int16", "int32"])
def test_no_synapses_beyond_the_one_cta_kernel(dtb, delivery, wfmt):
    tb = ng.make_tables(dict(ng.load_config("c2_multi_voxel_1m"), wfmt=wfmt, gain={"default": 1.3}), n_neurons=9001,
                        n_vox=3, K=0)
    d = ng.oracle_inputs(tb, ng.host_pull(tb), wfmt=wfmt)
    d["w_ext"] = 8 * 65536
    net = edge._net_from_dict(dtb, d, delivery)
    ref = oracle.OracleNet(d, "f32")
    spikes = edge._same_run(net, ref, [1, 40, 120])
    assert spikes > 0
    assert net.counters() == (0, spikes, 161)
    net.load_state(net.save_state())
    edge._same_run(net, ref, [30])


@pytest.mark.parametrize("delivery", ["bins", "queue"])
@pytest.mark.parametrize("check", ["test_network_without_synapses", "test_one_neuron_network", "test_spike_log_too_small",
                                   "test_timed_and_profiled_steps_match_the_oracle"])
def test_edge_cases(dtb, check, delivery):
    getattr(edge, check)(dtb, delivery)


@pytest.mark.parametrize("mode", [0, 1])
def test_both_schedules_in_bins(dtb, mode):
    edge.test_both_schedules_match_the_oracle(dtb, "bins", mode)


def test_wide_voxel_in_bins(dtb):
    edge.test_voxel_wider_than_the_delivery_window(dtb, "bins")


@pytest.mark.parametrize("wfmt", ["int16", "int32"])
def test_row_of_more_than_255_items_in_bins(dtb, wfmt):
    edge.test_row_longer_than_255_work_items(dtb, "bins", wfmt)


@pytest.mark.parametrize("wfmt", ["int16", "int32"])
def test_full_event_queue_in_bins(dtb, wfmt):
    parity.test_queue_overflow_spills_exactly(dtb, "bins", 1024, BIN_CAPACITY, wfmt)


@pytest.mark.parametrize("wfmt", ["int16", "int32"])
def test_bin_counters_cannot_wrap(dtb, wfmt):
    parity.test_event_counters_cannot_wrap(dtb, "bins", wfmt)


def test_ring_diagnostics_in_bins(dtb):
    parity.test_ring_diagnostics_match_dense_view(dtb, "bins")


@pytest.mark.parametrize("wfmt", ["int32", "int16"])
def test_several_tiles_in_bins(dtb, wfmt):
    parity.test_multivoxel_tiles_and_ragged_tail(dtb, wfmt, "bins")


def test_checkpoint_in_bins(dtb):
    parity.test_checkpoint_and_hyperparams(dtb, "bins")


@pytest.mark.slow
def test_one_second_in_bins(dtb):
    golden.test_c2_one_second_bit_exact("bins")
