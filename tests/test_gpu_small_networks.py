"""Networks of at most 3,072 neurons, whose steps run in one CTA: against the
C oracle at the edges of that path (one neuron, a full and an overfull block,
many small voxels, a hub row of several work items, every weight format, four
channels, the OU drive, a call of more steps than one launch takes), and the
hemodynamics and spike log against the general kernels on the same network."""
import numpy as np
import pytest

import oracle
from helpers import custom_net, params_row

pytestmark = pytest.mark.gpu
OU = dict(mu=0.1, sigma=0.15, tau=5.0)


def _inputs(n, voxel, n_ch, wfmt, hub=False):
    rng = np.random.default_rng(n + voxel)
    K = 20
    starts = np.append(np.arange(0, n, voxel), n).astype(np.int64)
    nv = len(starts) - 1
    rows = np.stack([params_row(g=(0.002 * f, 0.00002, 0.01, 0.0005)) for f in rng.uniform(1.0, 1.7, nv)])
    pre = rng.integers(0, n, (n, K))
    if hub:
        pre[:, 0] = 5  # neuron 5 has every neuron as a target
    w, kind, shift = {"int16": (rng.integers(150, 2500, (n, K)).astype(np.int16), oracle.W_INT16, 4),
                      "int32": (rng.integers(2000, 40000, (n, K)).astype(np.int32), oracle.W_INT32, 0),
                      "bf16": ((rng.uniform(0.05, 0.6, (n, K)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16),
                               oracle.W_BF16, 0),
                      "int8": (rng.integers(1, 121, (n, K)).astype(np.int8), oracle.W_INT8, 8)}[wfmt]
    d = custom_net(n, pre, rng.integers(0, n_ch, (n, K)), w, rows, voxel_start=starts,
                   delay_vv=rng.integers(1, 6, (nv, nv)), d_max=5, n_ch=n_ch, nu_ext=2000.0, w_ext=2 * 65536,
                   wfmt=kind, wshift=shift)
    if wfmt == "int8":  # with a power-of-two scale per source
        d["pre_shift"] = rng.integers(0, 4, n).astype(np.uint8)
    return d


def _net(dtb, d, wfmt, **kw):
    n, K = d["n"], d["K"]
    order = np.argsort(d["pre"].ravel(), kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(d["pre"].ravel(), minlength=n))
    tgt = np.repeat(np.arange(n, dtype=np.int64), K)
    word = (tgt[order] | (d["cls"].ravel()[order].astype(np.int64) << 30)).astype(np.uint32)
    csr = (row_ptr, word, np.ascontiguousarray(d["w"].ravel()[order])) + ((d["pre_shift"],) if "pre_shift" in d else ())
    return dtb.Network(n=n, voxel_start=d["voxel_start"], vparams=d["vparams"], delay_vv=d["delay_vv"],
                       d_max=d["d_max"], csr=csr, wfmt=wfmt,
                       wshift=d["wshift"], n_ch=d["n_ch"], dt=d["dt"], nu_ext=d["nu_ext"], w_ext=d["w_ext"],
                       seed=d["seed"], init_seed=d["init_seed"], bold=d["bold"], **kw)


@pytest.mark.parametrize("n,voxel,n_ch,wfmt,hub,ou", [(1, 1, 2, "int16", False, False), (1024, 1024, 2, "int16", True, False),
                                                      (1025, 9, 2, "int32", False, True), (3072, 2, 4, "bf16", False, False),
                                                      (2999, 500, 4, "int32", True, True), (2048, 341, 2, "int8", False, False)])
@pytest.mark.parametrize("delivery", ["ring", "bins"])
def test_small_networks_match_the_oracle(n, voxel, n_ch, wfmt, hub, ou, delivery):
    from paper_2308_01241_gb300 import dtb

    d = _inputs(n, voxel, n_ch, wfmt, hub)
    if ou:
        d["ou"] = OU
    net = _net(dtb, d, wfmt, delivery=delivery, ou=OU if ou else None, bold_every=50)
    general = _net(dtb, d, wfmt, delivery="queue", event_queue_capacity=100000, ou=OU if ou else None, bold_every=50)
    ref = oracle.OracleNet(d, "f32")
    total = 0
    for k in (1, 2, 47, 250):
        rids, roff = ref.run(k)
        for x in (net, general):
            x.step(k)
            ids, off = x.get_spikes()
            np.testing.assert_array_equal(off, roff)
            np.testing.assert_array_equal(ids, rids)
        np.testing.assert_array_equal(net.get_bold_samples(), general.get_bold_samples())
        total += len(rids)
    assert total > 0
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
    for a, b in zip(net.get_bold(), general.get_bold()):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(net.voxel_spikes(), general.voxel_spikes())
    assert net.counters() == general.counters() == (ref.events(), total, 300)
    if ou:
        np.testing.assert_array_equal(net.get_ou(), ref.get_ou())


def test_a_long_call_and_the_other_step_calls():
    from paper_2308_01241_gb300 import dtb

    d = _inputs(900, 300, 2, "int16")
    net = _net(dtb, d, "int16")
    ref = oracle.OracleNet(d, "f32")
    for how, k in (("step", 4500), ("timed", 40), ("step", 3), ("profile", 20), ("step", 61)):
        {"step": net.step, "timed": net.step_timed, "profile": net.profile_steps}[how](k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
