"""Networks created while torch's current stream still has work queued: on blocks of
the caching allocator that are free again for the next request, and on the device
arrays of the synapse table.  Rasters and state against the C oracle."""
import numpy as np
import pytest

import oracle
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


def _busy(torch):
    """Some tens of milliseconds of work on the current stream."""
    a = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
    for _ in range(40):
        a = (a @ a).clamp_(-1, 1)


@pytest.mark.parametrize("delivery", ["ring", "queue"])
@pytest.mark.parametrize("side", [False, True])
def test_creation_waits_for_queued_work(delivery, side):
    import torch

    from paper_2308_01241_gb300 import dtb

    tb = ng.make_tables(dict(ng.load_config("c2_multi_voxel_1m"), gain={"default": 1.35}), n_neurons=20011, n_vox=5,
                        K=100)
    pull = ng.host_pull(tb)
    host = dtb.host_csr(tb, pull)
    want = [torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda() for a in host]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ref = oracle.OracleNet(ng.oracle_inputs(tb, pull), "f32")
    rids, roff = ref.run(120)
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
        scratch = [torch.empty(24 << 20, dtype=torch.uint8, device="cuda") for _ in range(12)]
        csr = [torch.zeros_like(a) for a in want]
        _busy(torch)
        for a in scratch:
            a.fill_(255)
        del a, scratch  # free for the library's buffers, with the fills still to run
        for a, b in zip(csr, want):
            a.copy_(b)
        net = dtb.from_tables(tb, csr, delivery=delivery)
        net.step(120)
    ids, off = net.get_spikes()
    np.testing.assert_array_equal(off, roff)
    np.testing.assert_array_equal(ids, rids)
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
