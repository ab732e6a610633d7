"""The counters' test hook says so where the layout in use keeps no counters."""
import pytest

from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delivery,kw,counters", [
    ("ring", {}, False), ("queue", {}, False), ("bins", {}, False),
    ("queue", dict(event_queue_capacity=5000), True), ("bins", dict(bin_capacity=5000), True)])
def test_hook_needs_counters(delivery, kw, counters):
    from paper_2308_01241_gb300 import dtb

    tb = ng.make_tables(ng.load_config("c1_single_voxel_1k"))  # 1,000 neurons: the ring, unless a capacity is given
    net = dtb.from_tables(tb, dtb.host_csr(tb, ng.host_pull(tb)), delivery=delivery, **kw)
    if counters:
        net.test_preset_counters(1 << 32)
        return
    with pytest.raises(dtb.DtbError) as e:
        net.test_preset_counters(1 << 32)
    assert e.value.code == dtb.DTB_ESTATE
