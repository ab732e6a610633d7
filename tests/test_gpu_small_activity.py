"""A small network whose activity rises and falls between calls, so that its steps run
in one CTA, with the general kernels and in one CTA again: every call against the C
oracle; and at 245 Hz a call takes no longer than with the general kernels (which a
queue capacity of the caller's asks for)."""
import time

import numpy as np
import pytest

import oracle
from test_gpu_small_rows import _case, _net

pytestmark = pytest.mark.gpu


def _busy_case():
    d, csr = _case(3000, 200, 0, 0)
    d["w_ext"] = 8 * 65536
    return d, csr


def test_activity_that_changes_between_calls():
    d, csr = _busy_case()
    net, ref = _net(d, csr, delivery="ring"), oracle.OracleNet(d, "f32")
    loud = d["vparams"][:, 6:10].copy()
    quiet = loud.copy()
    quiet[:, :2] *= 0.02
    spikes = []
    for k, g in ((300, loud), (150, loud), (33, quiet), (400, quiet), (60, quiet), (40, loud), (250, loud), (70, loud)):
        net.set_hyperparams(g)
        ref.set_g(g)
        net.step(k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
        spikes.append(len(ids) / k)
    assert max(spikes) > 60 and min(spikes) < 1  # the line lies near 28 spikes a step
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
    assert net.counters()[0] == ref.events()
    blob = net.save_state()
    for _ in range(2):  # a restored state has no last call to go by
        net.load_state(blob)
        net.step(90)
        got = net.get_spikes()
    rids, roff = ref.run(90)
    np.testing.assert_array_equal(got[0], rids)
    np.testing.assert_array_equal(got[1], roff)


def test_high_rates_are_not_slower():
    d, csr = _busy_case()
    us = []
    for kw in (dict(delivery="ring"), dict(delivery="queue", event_queue_capacity=200_000)):
        net = _net(d, csr, **kw)
        net.step(1000)
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            net.step(500)
            best = min(best, time.perf_counter() - t0)
        us.append(best / 500 * 1e6)
    assert us[0] < 1.3 * us[1], us
