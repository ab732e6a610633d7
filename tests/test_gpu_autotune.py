"""dtb_autotune times the shapes in use, which need not be on its list, beside the
listed ones (46 runs in all, and one to warm up), and leaves a network whose steps
run in one CTA as it is; the steps that follow are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2308_01241_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shapes,runs", [(20_011, (2, 0, 5), 47), (20_011, (2, 0, 1), 46), (1_000, None, 0)])
def test_the_shapes_in_use_are_timed(n, shapes, runs):
    from paper_2308_01241_gb300 import dtb

    name = "c1_single_voxel_1k" if n == 1000 else "c2_multi_voxel_1m"
    tb = ng.make_tables(ng.load_config(name), n_neurons=n, n_vox=1 if n == 1000 else 5, K=60)
    pull = ng.host_pull(tb)
    net = dtb.from_tables(tb, dtb.host_csr(tb, pull))
    if shapes:
        net.set_shapes(*shapes)
    net.step(10)
    chosen = tuple(net.autotune(3).values())
    assert net.counters()[2] == 10 + 3 * runs
    listed = [(s, u, d) for s in (2, 3, 4) for u in (0, 1, 2) for d in (1, 2, 4, 6, 8)]
    assert chosen in listed + [shapes] if shapes else chosen[0] == 2
    assert net.get_spikes()[0].size == 0 or runs  # the log of a network that took no steps is empty
    net.reset()
    net.step(120)
    ids, off = net.get_spikes()
    rids, roff = oracle.OracleNet(ng.oracle_inputs(tb, pull), "f32").run(120)
    np.testing.assert_array_equal(off, roff)
    np.testing.assert_array_equal(ids, rids)
