"""Performance cases: the work that users of this framework have it do.

Each case is one call, or the short sequence of calls, that a program repeats:
a chunk of simulation steps with its raster and BOLD read back, one cycle of
data assimilation, one kernel-level call on device buffers, one pass of the
learned surrogate.  Sizes and options are those of the repository's own
configurations, studies, tests and benchmark, from the 1,000-neuron single
voxel to the largest network that fits the card three times over.

Inputs are made from the seed alone: the voxel structure, the synapses, the
drive and the initial state of a network all change with it.  Networks are
settled before the call, so that the steps run at their operating point.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2308_01241_gb300 import dtb, netgen
from paper_2308_01241_gb300.surrogate_mlp import MLP

DEVICE = "cuda:0"
DT_S = 1e-4          # one step, seconds of biological time
SETTLE = 2500        # steps after a reset until the rate has settled
OU = {"mu": 0.0, "sigma": 0.15, "tau": 5.0}
MLP_IN, MLP_WIDTH, MLP_DEPTH, MLP_OUT = 12, 256, 3, 6
LARGEST = 5_000_000  # neurons, in-degree 500


def _step(name, n, voxels, K, fmt, delivery, rate, steps, channels=2, ou=False):
    return {"name": name, "kind": "step", "n": n, "voxels": voxels, "K": K, "fmt": fmt, "delivery": delivery,
            "rate": rate, "steps": steps, "channels": channels, "ou": ou}


def listed():
    return [
        # the single-voxel configuration for its 1,000 steps, with the default
        # delivery: the smallest network, all launch latency
        _step("voxel_1k", 1_000, 1, 100, "int16", "ring", 15, 1000),
        # a ragged mid-size network with every optional part on: one channel
        # per receptor, the Ornstein-Uhlenbeck drive, the event-queue delivery
        _step("ragged_200k_ou", 200_003, 24, 100, "int32", "queue", 15, 200, channels=4, ou=True),
        # the 64-voxel, 1M-neuron configuration: 32-bit weights
        _step("voxels64_1m_int32", 1_000_000, 64, 500, "int32", "bins", 15, 200),
        # the precision study's 2M-neuron network with bfloat16 weights
        _step("precision_2m_bf16", 2_000_000, 200, 500, "bf16", "bins", 15, 200),
        # the in-degree sweep's dense end: 1,000 inputs per neuron, 8-bit weights
        _step("indegree1000_1500k", 1_500_000, 150, 1000, "int8", "bins", 15, 150),
        # the large-scale configuration's structure at its lowest and highest
        # operating point: the benchmark's workload
        _step("large_5m_7hz", LARGEST, 500, 500, "int16", "bins", 7, 100),
        _step("large_5m_30hz", LARGEST, 500, 500, "int16", "bins", 30, 100),
        # one cycle of the assimilation of a merged ensemble: 2 groups of 6
        # members and a hidden target each, predict + analysis + re-sampling
        {"name": "assimilate_2x7", "kind": "assimilate", "groups": 2, "members": 6, "neurons": 60_000, "voxels": 25,
         "steps": 2000},
        # the spike compaction alone on one step's bits of the 20M-neuron network
        {"name": "compact_20m", "kind": "compact", "n": 20_000_000, "rate": 15},
        # the analysis alone: 2,000 voxels, 128 members
        {"name": "enkf_2000x128", "kind": "enkf", "columns": 2000, "members": 128},
        # the surrogate's prediction of 122 members of 49 voxels
        {"name": "mlp_predict_5978", "kind": "mlp_forward", "batch": 5978},
        # the surrogate's training: four Adam steps on batches of 4,096
        {"name": "mlp_train_4096", "kind": "mlp_train", "batch": 4096, "batches": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    u = rng.random()
    if u < 0.6:
        n = _log_int(rng, 1_000, LARGEST)
        if n < 20_000:
            voxels, K = 1, rng.choice([50, 100, 150])
            delivery = rng.choice(["ring", "ring", "queue", "bins"])
        else:
            voxels = max(2, n // rng.choice([10_000, 16_000]))
            K = rng.choice([100, 200, 300, 500, 700, 1000])
            while n * K > LARGEST * 500:
                K = max(100, K // 2)
            delivery = "bins" if n > 1_000_000 else rng.choice(["bins", "bins", "queue", "ring"])
        fmt = rng.choice(["int16", "int16", "int32", "bf16", "int8"])
        return {"kind": "step", "n": n, "voxels": voxels, "K": K, "fmt": fmt, "delivery": delivery,
                "rate": rng.choice([7, 15, 30]), "steps": rng.randint(33, 100),
                "channels": 4 if rng.random() < 0.15 else 2, "ou": rng.random() < 0.15}
    if u < 0.68:
        return {"kind": "assimilate", "groups": rng.randint(1, 3), "members": rng.randint(2, 8),
                "neurons": _log_int(rng, 20_000, 80_000), "voxels": rng.randint(12, 60), "steps": rng.randint(300, 900)}
    if u < 0.78:
        return {"kind": "compact", "n": _log_int(rng, 1_000, 20_000_000), "rate": rng.choice([7, 15, 30])}
    if u < 0.86:
        return {"kind": "enkf", "columns": _log_int(rng, 49, 7000), "members": rng.randint(8, 300)}
    if u < 0.94:
        return {"kind": "mlp_forward", "batch": _log_int(rng, 300, 65_536)}
    return {"kind": "mlp_train", "batch": _log_int(rng, 500, 8_192), "batches": rng.randint(1, 4)}


# ----------------------------------------------------------------------------- networks
def _config(case, seed):
    """The repository's configuration for the case's structure, seeded, and its conductances [4]."""
    if case["voxels"] == 1:
        cfg = netgen.load_config("c1_single_voxel_1k")
        scale, gain = 100.0 / case["K"], cfg["gain"]["default"]
    else:
        cfg = netgen.load_config("c2_multi_voxel_1m" if case["fmt"] == "int32" else "c3_large_20m")
        # another in-degree keeps the mean recurrent input, as in the in-degree sweep
        scale, gain = 500.0 / case["K"], netgen.gain_for(cfg, case["rate"])
    cfg["w_ext"] = int(round(cfg["w_ext"] / scale))
    cfg["seeds"] = {k: 16 * int(seed) + i for i, k in enumerate(("net", "drive", "init", "vox"))}
    g = np.asarray(cfg["neuron"]["g"]) * scale
    g[:2] *= gain
    return cfg, g


def _synapses(tb, case, seed):
    """Device synapse table in the case's weight format and its weight shift."""
    if case["fmt"] == "int8":
        csr, shift = netgen.device_csr_int8(tb, device=DEVICE), 0
    else:
        csr, shift = netgen.device_csr(tb, case["fmt"], device=DEVICE), 4 if case["fmt"] == "int16" else 0
    if case["channels"] == 4:
        # excitatory synapses on AMPA or NMDA, inhibitory ones on GABAa or GABAb,
        # by source and target (a row's synapses come in no fixed order)
        row_ptr, word = csr[:2]
        src = torch.repeat_interleave(torch.arange(tb.n, device=DEVICE, dtype=torch.int32), row_ptr.diff())
        pick = ((word & 0x3FFFFFFF) * 40503 + src * 30011 + int(seed) % 65536) >> 9 & 1
        cls = ((word >> 30) & 3) * 2 + pick
        csr = (row_ptr, (word & 0x3FFFFFFF) | (cls << 30)) + tuple(csr[2:])
    return csr, shift


def _prepare_step(case, seed):
    cfg, g = _config(case, seed)
    tb = netgen.make_tables(cfg, n_neurons=case["n"], n_vox=case["voxels"], K=case["K"])
    csr, shift = _synapses(tb, case, seed)
    vp = tb.vparams(1.0)
    vp[:, 6:10] = g
    room = int(case["n"] * case["steps"] * DT_S * 150) + (1 << 16)  # ids at 150 Hz
    net = dtb.Network(n=tb.n, voxel_start=tb.voxel_start, vparams=vp, delay_vv=tb.delay_vv, d_max=tb.d_max, csr=csr,
                      wfmt=case["fmt"], wshift=shift, n_ch=case["channels"], dt=float(cfg["dt"]),
                      nu_ext=float(cfg["nu_ext"]), w_ext=cfg["w_ext"], seed=cfg["seeds"]["drive"],
                      init_seed=cfg["seeds"]["init"], bold=cfg["bold"], bold_every=8000, log_capacity=room,
                      delivery=case["delivery"], ou=OU if case["ou"] else None, device=DEVICE)
    net.step(SETTLE)
    return {"kind": "step", "net": net, "steps": case["steps"], "whole": case["n"] <= 250_000,
            "ids": torch.zeros(room, dtype=torch.int32, pin_memory=True).numpy(),
            "off": torch.zeros(case["steps"] + 1, dtype=torch.int64, pin_memory=True).numpy()}


def _run_step(s):
    net = s["net"]
    net.step(s["steps"])
    net.get_spikes(ids_out=s["ids"], off_out=s["off"])  # off[-1] ids of the program's own buffer
    y, hemo = net.get_bold()
    out = {"ids": s["ids"], "off": s["off"], "bold": y, "hemodynamics": hemo, "voxel_spikes": net.voxel_spikes()}
    if s["whole"]:  # a network this small is followed in full
        V, j, ref, _, t = net.get_state(with_ring=False)
        out.update(V=V, j=j, ref=ref, t=t)
    return out


def _prepare_assimilate(case, seed):
    cfg = netgen.load_config("c4_ensemble")
    # the groups' sizes stay; synapses, drive, initial state, prior and perturbations are the seed's
    cfg["seeds"].update({k: 16 * int(seed) + i for i, k in enumerate(("net", "drive", "init", "prior", "enkf"))})
    V, N, T = case["voxels"], case["neurons"], case["steps"]
    tb, lay = netgen.make_ensemble_tables(cfg, case["groups"], case["members"], (V - 5, V + 5),
                                          (N - N // 6, N + N // 6))
    csr = netgen.device_csr(tb, cfg["wfmt"], device=DEVICE)
    base = tb.vparams(1.0)
    net = dtb.Network(n=tb.n, voxel_start=tb.voxel_start, vparams=base, delay_vv=tb.delay_vv, d_max=tb.d_max, csr=csr,
                      wfmt=cfg["wfmt"], wshift=4, n_ch=int(cfg["n_ch"]), dt=float(cfg["dt"]),
                      nu_ext=float(cfg["nu_ext"]), w_ext=int(cfg["w_ext"]), seed=cfg["seeds"]["drive"],
                      init_seed=cfg["seeds"]["init"], bold=cfg["bold"], bold_every=T, delivery="bins",
                      log_capacity=1 << 16, device=DEVICE)
    # column = voxel of a group: its copies in the members, observed in the hidden target
    M = case["members"]
    vox = np.concatenate([np.stack([o + np.arange(k) for o, k in copies], 1) for copies in lay.net_vox])
    prior = cfg["prior"]
    rng = np.random.default_rng(cfg["seeds"]["prior"])
    theta = prior["log_gain_mean"] + prior["log_gain_sd"] * rng.standard_normal(vox.shape)
    gain = np.ones(tb.nv)
    gain[vox] = np.exp(theta)
    g = base[:, 6:10].copy()
    g[:, :2] *= gain[:, None]
    net.set_hyperparams(g)
    net.step(T)  # BOLD away from rest
    asm = dtb.Assimilation(net, vox[:, :M], theta[:, :M], base[:, 6:10], T, target_voxel=vox[:, M],
                           obs_sd_rel=cfg["enkf"]["obs_sd_rel"], inflation=cfg["enkf"]["inflation"],
                           seed=cfg["seeds"]["enkf"])
    return {"kind": "assimilate", "net": net, "asm": asm}


def _run_assimilate(s):
    theta, hx, y = s["asm"].assimilate(1)
    return {"theta": theta, "hx": hx, "y": y, "voxel_spikes": s["net"].voxel_spikes()}


# ----------------------------------------------------------------------------- kernel-level calls
def _prepare_compact(case, seed):
    n = case["n"]
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    words = -(-n // 1024) * 32
    fired = torch.rand(words * 32, generator=gen, device=DEVICE) < case["rate"] * DT_S
    fired[n:] = False
    weight = (torch.ones(32, dtype=torch.int64, device=DEVICE) << torch.arange(32, device=DEVICE))
    bits = (fired.view(words, 32).to(torch.int64) * weight).sum(1)
    bits = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits).to(torch.int32)
    return {"kind": "compact", "n": n, "bits": bits, "ids": torch.zeros(n, dtype=torch.int32, device=DEVICE),
            "count": torch.zeros(1, dtype=torch.int32, device=DEVICE)}


def _run_compact(s):
    dtb.dtb_spike_compact(s["bits"], s["n"], s["ids"], s["count"], torch.cuda.current_stream().cuda_stream)
    return {"ids": s["ids"], "count": s["count"]}


def _enkf_inputs(case, seed):
    C, M = case["columns"], case["members"]
    rng = np.random.default_rng(int(seed))
    theta = 0.18 + 0.08 * rng.standard_normal((C, M))
    hx = 0.02 + 0.05 * theta + 0.002 * rng.standard_normal((C, M))  # BOLD of the members
    y = hx.mean(1) + 0.004 * rng.standard_normal(C)
    sd = 0.02 * np.abs(y)
    eps = rng.standard_normal((C, M))
    return [a.astype(np.float32) for a in (theta, hx, y, sd, eps)]


def _prepare_enkf(case, seed):
    return {"kind": "enkf", "in": [torch.from_numpy(a).to(DEVICE) for a in _enkf_inputs(case, seed)]}


def _run_enkf(s):
    prior, hx, y, sd, eps = s["in"]
    theta = prior.clone()  # the analysis is in place and the prior is kept
    dtb.dtb_enkf_analysis(theta, hx, y, sd, eps, inflation=1.03, stream=torch.cuda.current_stream().cuda_stream)
    return theta


# ----------------------------------------------------------------------------- the learned surrogate
def _mlp_inputs(case, seed):
    """Parameters, standardised inputs and targets (float32, host)."""
    rng = np.random.default_rng(int(seed))
    sizes = [MLP_IN] + [MLP_WIDTH] * MLP_DEPTH + [MLP_OUT]
    params = [((rng.standard_normal((a, b)) * np.sqrt(2.0 / a)).astype(np.float32),
               (0.05 * rng.standard_normal(b)).astype(np.float32)) for a, b in zip(sizes[:-1], sizes[1:])]
    rows = case["batch"] * case.get("batches", 1)
    x = rng.standard_normal((rows, MLP_IN)).astype(np.float32)
    t = np.tanh(x[:, :MLP_OUT] + 0.5 * x[:, MLP_OUT:2 * MLP_OUT]) + 0.1 * rng.standard_normal((rows, MLP_OUT))
    return params, x, t.astype(np.float32)


def _prepare_mlp(case, seed):
    params, x, t = _mlp_inputs(case, seed)
    mlp = MLP(params, MLP_IN, MLP_WIDTH, MLP_DEPTH, MLP_OUT, max_batch=case["batch"])
    B = case["batch"]
    dx, dt = (torch.from_numpy(a).to(DEVICE) for a in (x, t))
    return {"kind": case["kind"], "mlp": mlp, "x": list(dx.split(B)), "t": list(dt.split(B)),
            "y": torch.zeros((B, MLP_OUT), device=DEVICE)}


def _run_mlp_forward(s):
    s["mlp"].forward(s["x"][0], s["y"], torch.cuda.current_stream().cuda_stream)
    return s["y"]


def _run_mlp_train(s):
    stream = torch.cuda.current_stream().cuda_stream
    loss = [s["mlp"].train_step(x, t, 1e-3, stream) for x, t in zip(s["x"], s["t"])]
    return {"loss": loss, "params": s["mlp"].params()}


# ----------------------------------------------------------------------------- the cases' functions
_PREPARE = {"step": _prepare_step, "assimilate": _prepare_assimilate, "compact": _prepare_compact,
            "enkf": _prepare_enkf, "mlp_forward": _prepare_mlp, "mlp_train": _prepare_mlp}
_RUN = {"step": _run_step, "assimilate": _run_assimilate, "compact": _run_compact, "enkf": _run_enkf,
        "mlp_forward": _run_mlp_forward, "mlp_train": _run_mlp_train}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["kind"]](state)


def work(case):
    """Bytes and operations that one pass cannot do without.

    A step reads and writes every neuron's V, four gating variables and
    refractory count (and OU current), writes its spike bit, and reads the
    outgoing synapses (target and weight) of the neurons that fire."""
    k = case["kind"]
    if k in ("step", "assimilate"):
        if k == "step":
            n, K, rate, ou = case["n"], case["K"], case["rate"], case["ou"]
            wb = {"int16": 2, "bf16": 2, "int32": 4, "int8": 1}[case["fmt"]]
        else:
            n, K, rate, ou, wb = case["groups"] * (case["members"] + 1) * case["neurons"], 200, 15, False, 2
        events = n * rate * DT_S * K
        per_step = n * (42.125 + (8 if ou else 0)) + events * (4 + wb) + 4 * n * rate * DT_S
        return {"bytes": case["steps"] * per_step, "flops": case["steps"] * (60.0 * n + events)}
    if k == "compact":
        return {"bytes": case["n"] / 8 + 4 * case["n"] * case["rate"] * DT_S + 4, "flops": case["n"] / 32}
    if k == "enkf":
        C, M = case["columns"], case["members"]
        return {"bytes": 4 * (4 * C * M + 2 * C), "flops": 14.0 * C * M}
    weights = MLP_IN * MLP_WIDTH + (MLP_DEPTH - 1) * MLP_WIDTH ** 2 + MLP_WIDTH * MLP_OUT
    B = case["batch"]
    if k == "mlp_forward":
        return {"bytes": 4.0 * B * (MLP_IN + MLP_OUT) + 2 * weights, "flops": 2.0 * B * weights}
    # forward, weight gradients, input gradients; Adam reads and writes weights and two moments
    return {"bytes": case["batches"] * (4.0 * B * (MLP_IN + MLP_OUT) + 24 * weights),
            "flops": case["batches"] * 6.0 * B * weights}


# ----------------------------------------------------------------------------- the same in 64 bits
def _exact_compact(case, seed):
    s = _prepare_compact(case, seed)
    shifts = torch.arange(32, device=DEVICE, dtype=torch.int32)
    on = ((s["bits"][:, None] >> shifts) & 1).reshape(-1)[: case["n"]]
    at = torch.nonzero(on).reshape(-1).to(torch.int32)
    ids = torch.zeros(case["n"], dtype=torch.int32, device=DEVICE)
    ids[: at.numel()] = at
    return {"ids": ids, "count": torch.tensor([at.numel()], dtype=torch.int32)}


def _exact_enkf(case, seed):
    theta, hx, y, sd, eps = (a.astype(np.float64) for a in _enkf_inputs(case, seed))
    a, h = theta - theta.mean(1, keepdims=True), hx - hx.mean(1, keepdims=True)
    m1 = theta.shape[1] - 1
    K = (a * h).sum(1) / m1 / ((h * h).sum(1) / m1 + sd * sd)
    post = theta + K[:, None] * (y[:, None] + sd[:, None] * eps - hx)
    mean = post.mean(1, keepdims=True)
    # the inflation is a 32-bit argument of the call
    return mean + float(np.float32(1.03)) * (post - mean)


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / 2.0 ** 0.5))


def _forward64(params, x):
    for k, (W, b) in enumerate(params):
        x = x @ W + b
        if k + 1 < len(params):
            x = _gelu(x)
    return x


def _mlp64(case, seed):
    params, x, t = _mlp_inputs(case, seed)
    d = lambda a: torch.from_numpy(a).to(DEVICE, torch.float64)  # noqa: E731
    return [(d(W), d(b)) for W, b in params], d(x), d(t)


def _exact_mlp_forward(case, seed):
    params, x, _ = _mlp64(case, seed)
    return _forward64(params, x)


def _exact_mlp_train(case, seed):
    params, X, T = _mlp64(case, seed)
    flat = [p.clone().requires_grad_(True) for pair in params for p in pair]
    m, v = [torch.zeros_like(p) for p in flat], [torch.zeros_like(p) for p in flat]
    losses = []
    for k, (x, t) in enumerate(zip(X.split(case["batch"]), T.split(case["batch"])), 1):
        loss = ((_forward64(list(zip(flat[::2], flat[1::2])), x) - t) ** 2).mean()
        losses.append(float(loss.detach()))
        grads = torch.autograd.grad(loss, flat)
        with torch.no_grad():
            for p, g, mp, vp in zip(flat, grads, m, v):
                mp.mul_(0.9).add_(0.1 * g)
                vp.mul_(0.999).add_(0.001 * g * g)
                p -= 1e-3 * (mp / (1 - 0.9 ** k)) / ((vp / (1 - 0.999 ** k)).sqrt() + 1e-8)
    out = [p.detach() for p in flat]
    return {"loss": losses, "params": list(zip(out[::2], out[1::2]))}


def exact(case, seed):
    """None for the simulated networks: a spiking network has no 64-bit
    counterpart (its rasters, sums and 32-bit state are defined bit by bit)."""
    f = {"compact": _exact_compact, "enkf": _exact_enkf, "mlp_forward": _exact_mlp_forward,
         "mlp_train": _exact_mlp_train}.get(case["kind"])
    return f(case, seed) if f else None
