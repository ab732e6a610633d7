"""Device memory of network creation, counted through the allocator hooks."""
import numpy as np
import pytest

import oracle
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


def _counting(dtb, monkeypatch, limit=None):
    """The binding's allocator with a count of live bytes, their peak, and a limit."""
    seen = {"live": 0, "peak": 0, "size": {}}

    class Counting(dtb._TorchAllocator):
        def _alloc(self, nbytes, ctx):
            if limit is not None and seen["live"] + nbytes > limit:
                return None
            p = super()._alloc(nbytes, ctx)
            if p:
                seen["size"][p] = nbytes
                seen["live"] += nbytes
                seen["peak"] = max(seen["peak"], seen["live"])
            return p

        def _free(self, p, ctx):
            seen["live"] -= seen["size"].pop(p)
            super()._free(p, ctx)

    monkeypatch.setattr(dtb, "_TorchAllocator", Counting)
    return seen


def _tables(wfmt):
    tb = ng.make_tables(dict(ng.load_config("c2_multi_voxel_1m"), wfmt=wfmt, gain={"default": 1.35}), n_neurons=20011,
                        n_vox=5, K=200)
    return tb, ng.host_pull(tb)


@pytest.mark.parametrize("delivery,bcap,wfmt", [("queue", 0, "int16"), ("bins", 20000, "int16"), ("queue", 0, "int32")])
def test_creation_needs_no_further_byte_per_synapse(monkeypatch, delivery, bcap, wfmt):
    """What creation frees again by its end is small next to the synapses: sums per
    neuron and counts per row, no buffer per synapse."""
    from paper_2308_01241_gb300 import dtb

    tb, pull = _tables(wfmt)
    csr = dtb.host_csr(tb, pull)
    seen = _counting(dtb, monkeypatch)
    net = dtb.from_tables(tb, csr, delivery=delivery, bin_capacity=bcap)
    assert seen["peak"] - seen["live"] < csr[1].size // 2
    ref = oracle.OracleNet(ng.oracle_inputs(tb, pull), "f32")
    net.step(150)
    ids, off = net.get_spikes()
    rids, roff = ref.run(150)
    assert len(rids) > 300
    np.testing.assert_array_equal(off, roff)
    np.testing.assert_array_equal(ids, rids)
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("delivery", ["queue", "bins"])
def test_a_layout_that_does_not_fit_gives_way(monkeypatch, delivery):
    """32-bit weights under an allocator with less room than the queue layout's
    packed records (8 bytes per synapse) need, but enough for a delay byte per
    synapse: the network is created and steps like the oracle.  Less room than the
    synapse table itself is still DTB_ENOMEM, with everything freed."""
    from paper_2308_01241_gb300 import dtb

    tb, pull = _tables("int32")
    csr = dtb.host_csr(tb, pull)
    nnz = csr[1].size
    seen = _counting(dtb, monkeypatch)
    net = dtb.from_tables(tb, csr, delivery="queue", log_capacity=1 << 20)
    packed = seen["peak"]
    net.close()
    assert seen["live"] == 0
    ref = oracle.OracleNet(ng.oracle_inputs(tb, pull), "f32")
    seen = _counting(dtb, monkeypatch, limit=packed - 4 * nnz)
    net = dtb.from_tables(tb, csr, delivery=delivery, log_capacity=1 << 20)
    assert seen["peak"] <= packed - 4 * nnz
    total = 0
    for k in (1, 40, 150):
        net.step(k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        total += len(rids)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
    assert total > 300
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
    net.close()
    seen = _counting(dtb, monkeypatch, limit=7 * nnz)
    with pytest.raises(dtb.DtbError) as e:
        dtb.from_tables(tb, csr, delivery=delivery, log_capacity=1 << 20)
    assert e.value.code == dtb.DTB_ENOMEM
    assert seen["live"] == 0
