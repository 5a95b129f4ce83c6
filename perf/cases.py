"""The work whose time this repository is measured by: cases over the public entry points.

A case is one call pattern of a user's program, on a network of the microcircuit's shape
(``workload.microcircuit``): stepping one network and reading its spikes and state ("step"),
many networks in one batch ("batch"), one surrogate-gradient evaluation ("grad"), stepping a
network held in the caller's own device memory ("noalloc") and delivering spike lists into the
ring buffers ("deliver").

``listed()`` names the measured cases, ``draw(rng)`` gives further ones of the same ranges,
``prepare`` builds what a program holds before the call, ``run`` makes one pass, ``work`` counts
the bytes and operations a pass cannot do without, and ``exact`` gives the same outputs from a
plain torch model in 64 bits that uses nothing of the library.
"""
import math

import numpy as np
import torch

import paper_1909_08665_gb300 as snn
import workload
from paper_1909_08665_gb300.autograd import microcircuit_rates

CKPT_EVERY = 100        # steps between the gradient's checkpoints, as its configuration sets
NOALLOC_RASTER = 1 << 22


def listed():
    return [
        # A controller in a closed loop: 1 ms of the 10 % network, its spikes read every time.
        # The smallest call; launches, synchronisations and copies count.
        {"name": "step_loop_1ms", "kind": "step", "scale": 0.1, "input": "poisson", "steps": 10},
        # The 10 % network for 100 ms: the repository's first configuration.
        {"name": "step_tenth_100ms", "kind": "step", "scale": 0.1, "input": "poisson", "steps": 1000},
        # One second of the full microcircuit, raster and state read: the headline workload.
        {"name": "step_full_1s", "kind": "step", "scale": 1.0, "input": "poisson", "steps": 10000},
        # The DC-driven variant at an odd size.
        {"name": "step_dc_odd", "kind": "step", "scale": 0.3717, "input": "dc", "steps": 1537},
        # The scaled-up network, 308,676 neurons and 1.2e9 synapses.
        {"name": "step_4x_100ms", "kind": "step", "scale": 4.0, "input": "poisson", "steps": 1000},
        # 64 networks of uneven size in one launch: a parameter study.
        {"name": "batch_64_100ms", "kind": "batch", "n": 64, "lo": 0.05, "hi": 0.25, "dc": False,
         "steps": 1000},
        # A handful of small networks, DC-driven ones among them, for a ragged number of steps.
        {"name": "batch_5_ragged", "kind": "batch", "n": 5, "lo": 0.013, "hi": 0.05, "dc": True,
         "steps": 257},
        # Fitting the population rates of the 10 % network over 200 ms, checkpoints every 100
        # steps and every segment re-run by the backward.
        {"name": "grad_200ms_ckpt", "kind": "grad", "scale": 0.1, "steps": 2000, "record": False},
        # The same over a short horizon on a smaller network, the trajectory recorded: the
        # horizon at which the gradient is a training signal.
        {"name": "grad_10ms", "kind": "grad", "scale": 0.05, "steps": 100, "record": True},
        # A real-time application that owns all device memory, 1 ms at a time.
        {"name": "noalloc_loop_1ms", "kind": "noalloc", "scale": 0.1, "steps": 10},
        # The same on the full microcircuit for 100 ms.
        {"name": "noalloc_full_100ms", "kind": "noalloc", "scale": 1.0, "steps": 1000},
        # Replaying long spike lists into the full network's ring buffers, and reading those.
        {"name": "deliver_20000", "kind": "deliver", "scale": 1.0, "spikes": 20000, "lists": 16,
         "tiling": 3},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "grad", "noalloc", "deliver"])
    if kind == "step":
        scale = round(_log(rng, 0.02, 4.0), 4)
        most = min(10000.0, 10000.0 / scale)            # neuron-steps of the largest listed case
        return {"kind": kind, "scale": scale, "input": rng.choice(["poisson", "poisson", "dc"]),
                "steps": int(_log(rng, 10, most))}
    if kind == "batch":
        lo = round(_log(rng, 0.013, 0.1), 4)
        return {"kind": kind, "n": int(_log(rng, 2, 64.99)), "lo": lo,
                "hi": round(min(0.25, lo * rng.uniform(1.5, 5.0)), 4),
                "dc": rng.random() < 0.5, "steps": int(_log(rng, 50, 1000))}
    if kind == "grad":
        return {"kind": kind, "scale": round(_log(rng, 0.02, 0.1), 4),
                "steps": int(_log(rng, 60, 2000)), "record": rng.random() < 0.5}
    if kind == "noalloc":
        return {"kind": kind, "scale": round(_log(rng, 0.02, 1.6), 4), "steps": int(_log(rng, 10, 1000))}
    scale = round(_log(rng, 0.1, 1.0), 4)
    return {"kind": kind, "scale": scale, "spikes": int(_log(rng, 25, min(20000.0, 70000.0 * scale))),
            "lists": rng.randint(1, 16), "tiling": 3}


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------
def _configs(case, seed):
    """The networks of a case: configuration dictionaries with their seeds."""
    if case["kind"] == "batch":
        cfgs = workload.batched_instances(case["n"], 7, case["lo"], case["hi"])
        if case["dc"]:
            cfgs = [workload.dc_variant(c) if k % 3 == 2 else c for k, c in enumerate(cfgs)]
        seeds = np.random.default_rng(seed).integers(1, 2**62, len(cfgs))
        return [dict(c, seed=int(s)) for c, s in zip(cfgs, seeds)]
    if case["kind"] == "grad":
        return [workload.microcircuit(case["scale"], 12345)]
    return [workload.microcircuit(case["scale"], 12345 + seed, case.get("input", "poisson"))]


def _grad_inputs(cfg, seed):
    """Projection scales, background rate, target rates and initial potentials: the connectome
    itself stays while its parameters are fitted."""
    rng = np.random.default_rng(seed)
    return (rng.uniform(0.95, 1.05, (8, 8)).astype(np.float32), np.float32(cfg["nu_bg"]),
            workload.target_rates(11 + seed), workload.random_membrane(cfg, seed))


def _raster_rows(case, cfgs):
    """Rows of the program's spike record: room for 16 Hz and for the first volley."""
    n = sum(workload.n_neurons(c) for c in cfgs)
    return int(16.0 * n * case["steps"] * 1e-4) + n // 2 + 64


def _record(raster, steps, ids):
    """The spikes of one pass into the program's record (-1 past the last one)."""
    m = min(steps.size, raster.shape[1])
    raster[0, :m], raster[1, :m] = steps[:m], ids[:m]
    raster[:, m:] = -1
    return raster


def prepare(case, seed):
    kind, cfgs = case["kind"], _configs(case, seed)
    stream = torch.cuda.current_stream()
    state = {"case": case}
    if kind == "batch":
        state["net"] = snn.MicrocircuitBatch(cfgs, stream=stream)
        state["raster"] = np.empty((2, _raster_rows(case, cfgs)), np.int32)
        return state
    u0 = None
    if kind == "grad":
        scales, nu, targets, u0 = _grad_inputs(cfgs[0], seed)
    net = state["net"] = snn.Microcircuit(cfgs[0], u0=u0, stream=stream)
    if kind == "step":
        state["raster"] = np.empty((2, _raster_rows(case, cfgs)), np.int32)
    elif kind == "grad":
        net.set_grad_trace_budget((4 << 30) if case["record"] else 0)
        state["start"] = net.save_state()
        state["scales"] = torch.from_numpy(scales).cuda()
        state["nu"] = torch.tensor(nu, device="cuda")
        state["targets"] = torch.from_numpy(targets).cuda()
    elif kind == "deliver":
        lists = [workload.random_spike_list(net.n, case["spikes"], 1000 * seed + k)
                 for k in range(case["lists"])]
        state["lists"] = torch.from_numpy(np.stack(lists).view(np.int32)).cuda()
    elif kind == "noalloc":
        row_ptr, words, wtab = net.export_network()
        u, i_syn, refr = net.state()
        net.close()
        d = {"row_ptr": row_ptr.view(np.int64), "words": words.view(np.int32),
             "wtab": wtab.reshape(-1), "u": u, "i_syn": i_syn, "refr": refr}
        d = {k: torch.from_numpy(v).cuda() for k, v in d.items()}
        zeros = lambda n, dtype: torch.zeros(n, dtype=dtype, device="cuda")  # noqa: E731
        d["ring"] = zeros(snn.RING_DEPTH * u.size, torch.int32)
        d["ras_step"], d["ras_id"] = zeros(NOALLOC_RASTER, torch.int32), zeros(NOALLOC_RASTER, torch.int32)
        d["ras_n"], d["status"] = zeros(1, torch.int32), zeros(1, torch.int32)
        d["counters"] = zeros(2, torch.int64)
        state.update(net=None, cfg=cfgs[0], bufs=d, t=0, stream=stream,
                     io=snn.SnnNoallocIO(ras_cap=NOALLOC_RASTER,
                                         **{k: v.data_ptr() for k, v in d.items()}))
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, net = state["case"], state["net"]
    kind = case["kind"]
    if kind == "step":
        net.step(case["steps"])
        steps, ids = net.read_spikes()
        u, i_syn, refr = net.state()
        return {"count": steps.size, "raster": _record(state["raster"], steps, ids),
                "u": u, "i_syn": i_syn, "refr": refr}
    if kind == "batch":
        net.step(case["steps"])
        spikes = [net.read_spikes(k) for k in range(len(net))]
        states = [net.state(k) for k in range(len(net))]
        out = {name: np.concatenate([s[k] for s in states])
               for k, name in enumerate(("u", "i_syn", "refr"))}
        out["count"] = np.array([s.size for s, _ in spikes])
        out["raster"] = _record(state["raster"], np.concatenate([s for s, _ in spikes]),
                                np.concatenate([i for _, i in spikes]))
        return out
    if kind == "grad":
        scales = state["scales"].detach().requires_grad_()
        nu = state["nu"].detach().requires_grad_()
        rates = microcircuit_rates(scales, nu, net, case["steps"], CKPT_EVERY, state["start"])
        loss = ((rates - state["targets"]) ** 2).mean()
        loss.backward()
        return {"rates": rates.detach(), "loss": loss.detach(), "d_scales": scales.grad, "d_nu": nu.grad}
    if kind == "noalloc":
        d = state["bufs"]
        d["ras_n"].zero_()
        snn.step_noalloc(state["cfg"], state["cfg"]["seed"], state["io"], state["t"], case["steps"],
                         state["stream"])
        state["t"] += case["steps"]
        # the raster's order within a step is unspecified; its spikes show in all of these
        return {k: d[k] for k in ("u", "i_syn", "refr", "ring", "ras_n", "counters")}
    for k in range(case["lists"]):
        net.deliver(state["lists"][k].data_ptr(), state["lists"].shape[1], k, case["tiling"])
    return {"ring": net.ring()}


def work(case):
    """Bytes: the 4-byte synaptic words of the spikes' rows (a mean rate of 6 Hz, the network's),
    the state read once and written once, the spikes and the state handed back.  Operations: about
    12 for a neuron's update and 2 for each synaptic event; the adjoint touches every synapse in
    every step."""
    kind = case["kind"]
    if kind == "batch":
        scales = [(case["lo"] + case["hi"]) / 2] * case["n"]
    else:
        scales = [case["scale"]]
    nbytes = flops = 0.0
    for s in scales:
        n = float(sum(workload.population_sizes(s)))
        row = workload.SYNAPSES_FULL / workload.N_FULL * min(1.0, s)
        ring = 4.0 * snn.RING_DEPTH * n
        if kind == "deliver":
            events = float(case["spikes"] * case["lists"]) * row
            nbytes += 4.0 * events + 2.0 * ring
            flops += 2.0 * events
            continue
        t = case["steps"]
        spikes = 6.0 * n * t * 1e-4
        nbytes += spikes * (4.0 * row + 8.0) + 2.0 * (12.0 * n + ring) + 12.0 * n
        flops += 12.0 * n * t + 2.0 * spikes * row
        if kind == "grad":                       # trace written and read once, rows read once
            nbytes += 2.0 * 5.0 * n * t + 4.0 * n * row
            flops += 2.0 * n * row * t + 16.0 * n * t
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same outputs from a plain model in 64 bits
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    m = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2          # the low 64 bits, as int64
        c0, c1, c2, c3 = (((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m)
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _f64(x):
    return torch.tensor(x, dtype=torch.float64, device="cuda")


def _round(x):
    return torch.sign(x) * torch.floor(x.abs() + 0.5)


def _network(cfg):
    """One network as its seed defines it: rows (target, delay, weight in 1/256 pA, unrounded base
    weight), sorted by source, and per-neuron tables."""
    sizes = torch.tensor(cfg["pop_sizes"], device="cuda")
    n, n_pop = int(sizes.sum()), len(cfg["pop_sizes"])
    pop = torch.repeat_interleave(torch.arange(n_pop, device="cuda"), sizes)
    k0, k1 = cfg["seed"] & 0xFFFFFFFF, cfg["seed"] >> 32
    thr = torch.floor(_f64(cfg["conn_prob"]) * cfg["conn_scale"] * 2.0**32).clamp(0, 2.0**32).long()
    z_w = torch.special.ndtri((torch.arange(128, device="cuda").double() + 0.5) / 128)
    base = (_f64(cfg["w_mean"])[..., None] + _f64(cfg["w_sd"])[..., None] * z_w) * cfg["w_scale"]
    weight = _round(base * _f64(cfg["proj_scale"])[..., None] * 256.0).long()
    z_d = torch.special.ndtri((torch.arange(256, device="cuda").double() + 0.5) / 256)
    delay = _round((_f64(cfg["d_mean"])[:, None] + _f64(cfg["d_sd"])[:, None] * z_d) / cfg["dt"]).clamp(1, 63)
    groups = torch.arange((n + 3) // 4, device="cuda")[None]
    rows, parts = max(1, (1 << 26) // n), []
    for lo in range(0, n, rows):
        j = torch.arange(lo, min(n, lo + rows), device="cuda")[:, None]
        zero = torch.zeros_like(j + groups)
        x = torch.stack(_philox(zero + j, zero + groups, zero + 1, zero, k0, k1), -1).reshape(j.shape[0], -1)[:, :n]
        hit = x < thr[pop[None], pop[j]]
        hit[torch.arange(j.shape[0], device="cuda"), j[:, 0]] = False
        src, tgt = hit.nonzero(as_tuple=True)
        src += lo
        zero = torch.zeros_like(src)
        y = _philox(src, tgt, zero + 2, zero, k0, k1)
        p, q, code = pop[tgt], pop[src], y[0] >> 25
        parts.append((src, tgt, delay[q, y[1] >> 24].long(), weight[p, q, code], base[p, q, code]))
        del x, hit, zero, y
    net = dict(zip(("src", "tgt", "delay", "w", "base"), (torch.cat(c) for c in zip(*parts))))
    lam = [cfg["nu_bg"] * k * cfg["dt"] / 1000.0 for k in cfg["k_ext"]]
    pois = torch.full((n_pop, 32), 1 << 32, device="cuda")      # DC: no count is ever reached
    for p in range(n_pop if cfg["input_mode"] == 0 else 0):
        term = cdf = math.exp(-lam[p])
        for m in range(32):
            if m:
                term = term * lam[p] / m
                cdf += term
            pois[p, m] = min(math.floor(cdf * 2.0**32), 1 << 32)
    i = torch.arange(n, device="cuda")
    bits = _philox(i, i * 0, i * 0 + 4, i * 0, k0, k1)[0] >> 8
    lo, hi = np.float32(cfg["u0_lo"]), np.float32(cfg["u0_hi"])
    p20 = cfg["tau_m"] / cfg["c_m"] * (1.0 - math.exp(-cfg["dt"] / cfg["tau_m"]))
    net.update(n=n, pop=pop, pois=pois[pop], k0=i * 0 + k0, k1=i * 0 + k1, local=i,
               u0=float(lo) + float(hi - lo) * (bits.float() * 2.0**-24),
               cdc=(p20 * _f64(cfg["i_dc"]) if cfg["input_mode"] == 1 else _f64(cfg["i_dc"]) * 0)[pop])
    return net


def _propagators(cfg):
    """P22, P21, P11 as the model fixes them: rounded once to 32 bits."""
    p22, p11 = math.exp(-cfg["dt"] / cfg["tau_m"]), math.exp(-cfg["dt"] / cfg["tau_syn"])
    p21 = cfg["tau_m"] * cfg["tau_syn"] / (cfg["c_m"] * (cfg["tau_m"] - cfg["tau_syn"])) * (p22 - p11)
    return [float(np.float32(v)) for v in (p22, p21, p11)]


def _simulate(cfgs, steps, u0=None, trace=False):
    """`steps` steps of the networks side by side.  Spikes are decided by the model's own 32-bit
    arithmetic (one rounding per operation); u and I are carried in 64 bits along that spike train."""
    nets = [_network(c) for c in cfgs]
    first = np.cumsum([0] + [m["n"] for m in nets])
    n, cfg = int(first[-1]), cfgs[0]
    cat = {k: torch.cat([m[k] for m in nets]) for k in ("pois", "k0", "k1", "local", "u0", "cdc", "delay", "w", "base", "pop")}
    src = torch.cat([m["src"] + int(f) for m, f in zip(nets, first)])
    cat["src"], cat["tgt"] = src, torch.cat([m["tgt"] + int(f) for m, f in zip(nets, first)])
    length = torch.bincount(src, minlength=n)
    start = torch.cumsum(length, 0) - length
    cell = cat["delay"] * n + cat["tgt"]
    p22, p21, p11 = _propagators(cfg)
    theta, w_ext = float(np.float32(cfg["theta"])), round(cfg["w_ext"] * 256.0)
    n_ref = round(cfg["t_ref"] / cfg["dt"])
    ring = torch.zeros(64, n, dtype=torch.int64, device="cuda")
    u, i_syn, refr = cat["u0"] if u0 is None else u0, torch.zeros(n, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda")
    u64, i64 = u.double(), i_syn.double()
    cdc32 = cat["cdc"].float()
    events, raster, seen = 0, [], []
    for t in range(steps):
        if t % 4 == 0:
            draws = _philox(cat["local"], cat["local"] * 0 + (t >> 2), cat["local"] * 0 + 3, cat["local"] * 0, cat["k0"], cat["k1"])
        count = (draws[t % 4][:, None] >= cat["pois"]).sum(1)
        acc = ring[t % 64] + w_ext * count
        ring[t % 64] = 0
        live = refr == 0
        refr = (refr - 1).clamp_min(0)
        v = torch.add(p22 * u, p21 * i_syn)
        u = torch.where(live, torch.where(cdc32 != 0, v + cdc32, v), 0.0)
        u64 = torch.where(live, p22 * u64 + p21 * i64 + cat["cdc"], 0.0)
        i_syn = torch.add(p11 * i_syn, acc.float() * 0.00390625)
        i64 = p11 * i64 + acc.double() / 256.0
        spk = u > theta
        if trace:
            seen.append((u.clone(), spk, live))
        ids = spk.nonzero()[:, 0]
        u[ids], u64[ids], refr[ids] = 0.0, 0.0, n_ref
        if ids.numel():
            ln = length[ids]
            pos = torch.repeat_interleave(start[ids] - (torch.cumsum(ln, 0) - ln), ln)
            pos += torch.arange(pos.numel(), device="cuda")
            ring.view(-1).index_add_(0, (cell[pos] + (t % 64) * n) % (64 * n), cat["w"][pos])
            events += pos.numel()
        raster.append(ids)
    ids = torch.cat(raster)
    at = torch.repeat_interleave(torch.arange(steps, device="cuda"), torch.tensor([r.numel() for r in raster], device="cuda"))
    return {"net": cat, "first": first, "n": n, "ring": ring, "u": u64, "i_syn": i64, "refr": refr, "ids": ids, "at": at,
            "events": events, "trace": seen}


def _exact_grad(case, seed):
    cfg = _configs(case, seed)[0]
    scales, nu, targets, u0 = _grad_inputs(cfg, seed)
    cfg = dict(cfg, proj_scale=scales.astype(np.float64).tolist(), nu_bg=float(nu))
    sim = _simulate([cfg], case["steps"], u0=torch.from_numpy(u0).cuda(), trace=True)
    net, n, steps = sim["net"], sim["n"], case["steps"]
    sizes, pop = _f64(cfg["pop_sizes"]), sim["net"]["pop"]
    seconds = steps * cfg["dt"] / 1000.0
    rates = (torch.bincount(pop[sim["ids"]], minlength=8).double() / (sizes * seconds)).requires_grad_()
    loss = ((rates - torch.from_numpy(targets).cuda()) ** 2).mean()
    loss.backward()
    gs = (rates.grad / (sizes * seconds))[pop]
    p22, p21, p11 = _propagators(cfg)
    theta = float(np.float32(cfg["theta"]))
    lam_i = torch.zeros(steps + 64, n, dtype=torch.float64, device="cuda")
    lam_u, live_next = torch.zeros_like(gs), torch.zeros(n, dtype=torch.bool, device="cuda")
    proj = pop[net["tgt"]] * 8 + pop[net["src"]]
    g_scales, w = torch.zeros(64, dtype=torch.float64, device="cuda"), net["w"].double() / 256.0
    for t in range(steps - 1, -1, -1):
        u, spk, live = sim["trace"][t]
        pull = lam_i.view(-1)[(net["delay"] + t) * n + net["tgt"]]
        ds = gs.clone().index_add_(0, net["src"], w * pull)
        hit = spk[net["src"]].nonzero()[:, 0]
        g_scales.index_add_(0, proj[hit], net["base"][hit] * pull[hit])
        lam_i[t] = p11 * lam_i[t + 1] + torch.where(live_next, p21 * lam_u, 0.0)
        slope = 1.0 / (1.0 + 10.0 * (u.double() - theta).abs()) ** 2
        lam_u = ds * slope + torch.where(live_next & ~spk, p22 * lam_u, 0.0)
        live_next = live
    per_nu = round(cfg["w_ext"] * 256.0) / 256.0 * _f64(cfg["k_ext"]) * cfg["dt"] / 1000.0
    return {"rates": rates.detach(), "loss": loss.detach(), "d_scales": g_scales.reshape(8, 8),
            "d_nu": (lam_i.sum(0) * per_nu[pop]).sum()}


def exact(case, seed):
    """None for the ring of a delivery (whole numbers) and for networks above the full size."""
    kind = case["kind"]
    if kind == "deliver" or case.get("scale", 0.0) > 2.0:
        return None
    if kind == "grad":
        return _exact_grad(case, seed)
    sim = _simulate(_configs(case, seed), case["steps"])
    out = {k: sim[k] for k in ("u", "i_syn", "refr")}
    if kind == "noalloc":
        out.update(ring=sim["ring"].reshape(-1), ras_n=_f64([sim["ids"].numel()]).int(),
                   counters=torch.tensor([sim["ids"].numel(), sim["events"]], device="cuda"))
        return out
    first = torch.from_numpy(sim["first"]).cuda()
    inst = torch.searchsorted(first, sim["ids"], right=True) - 1
    order = torch.argsort(inst, stable=True)
    raster = np.empty((2, _raster_rows(case, _configs(case, seed))), np.int32)
    out["raster"] = _record(raster, sim["at"][order].cpu().numpy(), (sim["ids"] - first[inst])[order].cpu().numpy())
    count = torch.bincount(inst, minlength=len(sim["first"]) - 1)
    out["count"] = count if kind == "batch" else int(count)
    return out
