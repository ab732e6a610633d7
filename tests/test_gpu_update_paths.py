"""The neuron update's branches against the C oracle, bit for bit: quads of
four neurons inside one voxel, across voxel boundaries (voxels of a few
neurons) and at the ragged end of the last tile; few and many Poisson
thresholds; with and without the OU current; two and four channels."""
import numpy as np
import pytest

import oracle
from helpers import custom_net, params_row

pytestmark = pytest.mark.gpu


def _net(dtb, d, delivery, ou=None):
    n, K = d["n"], d["K"]
    order = np.argsort(d["pre"].ravel(), kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(d["pre"].ravel(), minlength=n))
    tgt = np.repeat(np.arange(n, dtype=np.int64), K)
    word = (tgt[order] | (d["cls"].ravel()[order].astype(np.int64) << 30)).astype(np.uint32)
    return dtb.Network(n=n, voxel_start=d["voxel_start"], vparams=d["vparams"], delay_vv=d["delay_vv"],
                       d_max=d["d_max"], csr=(row_ptr, word, np.ascontiguousarray(d["w"].ravel()[order])),
                       wfmt="int32", wshift=0, n_ch=d["n_ch"], dt=d["dt"], nu_ext=d["nu_ext"], w_ext=d["w_ext"],
                       seed=d["seed"], init_seed=d["init_seed"], bold=d["bold"], delivery=delivery, ou=ou)


@pytest.mark.parametrize("delivery", ["ring", "queue", "bins"])
@pytest.mark.parametrize("n,voxel,nu_ext,n_ch,ou", [(1027, 5, 2000.0, 2, False), (4099, 1027, 2000.0, 2, False),
                                                     (2050, 7, 20000.0, 4, True), (5121, 513, 500.0, 2, True)])
def test_update_branches_match_the_oracle(n, voxel, nu_ext, n_ch, ou, delivery):
    from paper_2308_01241_gb300 import dtb

    rng = np.random.default_rng(n)
    K = 20
    starts = np.append(np.arange(0, n, voxel), n).astype(np.int64)
    nv = len(starts) - 1
    rows = np.stack([params_row(g=(0.002 * f, 0.00002, 0.01, 0.0005), t_ref=1.0 + 0.1 * (v % 20))
                     for v, f in enumerate(rng.uniform(0.8, 1.6, nv))])
    d = custom_net(n, rng.integers(0, n, (n, K)), rng.integers(0, n_ch, (n, K)),
                   rng.integers(2000, 40000, (n, K)).astype(np.int32), rows, voxel_start=starts,
                   delay_vv=rng.integers(1, 6, (nv, nv)), d_max=5, n_ch=n_ch, nu_ext=nu_ext,
                   w_ext=int(65536 * 2000.0 / nu_ext))
    cur = dict(mu=0.1, sigma=0.15, tau=5.0) if ou else None
    if ou:
        d["ou"] = cur
    net = _net(dtb, d, delivery, cur)
    ref = oracle.OracleNet(d, "f32")
    total = 0
    for k in (1, 45, 200):
        net.step(k)
        ids, off = net.get_spikes()
        rids, roff = ref.run(k)
        np.testing.assert_array_equal(off, roff)
        np.testing.assert_array_equal(ids, rids)
        total += len(ids)
    assert total > 100
    for a, b in zip(net.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)
    if ou:
        np.testing.assert_array_equal(net.get_ou(), ref.get_ou())
