"""Performance cases of the spiking-network engine: what its users run, through the public binding.

Every pass starts from the same point (a reset, a checkpoint, or a new net), so that repeated passes do
the same work; the seed of a case's inputs is the network's (its connectivity and its thalamic drive) or
that of the host's stimulus.  Kinds of pass:

  simulate   reset, run `steps` ms, read the neurons' state, the counters and, where the case says so,
             the raster and every synapse's weight and derivative
  step       one millisecond driven by host events, spike count and state read back (closed loop)
  window     reset, one end-to-end call: host events in, raster of the window out
  resume     explicit synapse lists: load a checkpoint, run, read raster and weights
  request    what a served request does: build a net, run it, read its raster, free it
  batch      reset and advance uneven independent nets together
"""
import math

import numpy as np

import paper_1310_8478_gb300 as eng
import workloads

# projection mixes: the benchmark's and the paper's (own column, first, second, third ring)
MIX = {"bench": (40, 30, 20, 10), "paper": (76, 12, 8, 4), "local": (100, 0, 0, 0)}


def _case(kind, gx, gy, npc, fanout, mix, steps, **more):
    c = dict(kind=kind, gx=gx, gy=gy, npc=npc, fanout=fanout, mix=mix, steps=steps, fp64=False, raster=False,
             weights=False, nets=1)
    c.update(more)
    return c


def listed():
    return [
        # an online loop (a controller, a body model): one column, one millisecond per call, host events in
        _case("step", 1, 1, 1250, 100, "local", 1, name="step"),
        # the one-column workload for its whole second, across the long-term update; everything read back
        _case("simulate", 1, 1, 1250, 100, "local", 1000, raster=True, weights=True, name="column"),
        # the same column in the double-precision physics mode
        _case("simulate", 1, 1, 1250, 100, "local", 200, fp64=True, raster=True, name="column_fp64"),
        # a user's own connectome (uneven rows, any target, any delay), continued from a checkpoint
        _case("resume", 2, 2, 1250, 100, "local", 100, raster=True, weights=True, name="resume"),
        # one served request: an 8x8 torus of the paper's columns, 200 ms, built for it and freed after it
        _case("request", 8, 8, 1000, 200, "paper", 200, raster=True, name="request"),
        # a stimulus-response trial on the paper's 16x16 torus: host events in, raster out
        _case("window", 16, 16, 1000, 200, "paper", 200, raster=True, name="window"),
        # a learning experiment: a second and a bit of the paper's 8x8 torus, then all weights
        _case("simulate", 8, 8, 1000, 200, "paper", 1010, weights=True, name="learning"),
        # the paper's 64x64 torus (4.1 M neurons, 819 M synapses) at its ~20 Hz
        _case("simulate", 64, 64, 1000, 200, "paper", 100, name="paper64"),
        # a busier net: 300 synapses per neuron, 7 to 8 % of the neurons firing each millisecond
        _case("simulate", 32, 32, 1000, 300, "paper", 200, name="busy"),
        # the benchmark torus at half its size (2.9 G synapses) over its onset, quiet to a quarter firing
        _case("simulate", 64, 32, 1250, 1125, "bench", 25, name="onset"),
        # the same columns in the run-away regime that fills their first second (1.4 G synapses)
        _case("simulate", 32, 32, 1250, 1125, "bench", 100, name="runaway"),
        # uneven independent nets advanced together: sides 1..16, fan-outs 100, 400 and 1125
        _case("batch", 16, 16, 1250, 1125, "bench", 50, nets=24, name="batch"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: any kind, columns of 300 to 1500 neurons, sides 1 to 64, 16 to 1125 synapses per neuron."""
    kind = rng.choice(["step", "simulate", "simulate", "simulate", "simulate", "resume", "request", "window", "batch"])
    npc = rng.choice([1000, 1250, rng.randint(300, 1500)])
    fanout = _log_int(rng, 16, 1125)
    side = {"step": 4, "resume": 3, "request": 10, "window": 20, "batch": 12, "simulate": 48}[kind]
    gx, gy = _log_int(rng, 1, side), _log_int(rng, 1, side)
    mix = "local" if gx * gy == 1 else rng.choice(["bench", "paper"])
    nets = rng.randint(3, 24) if kind == "batch" else 1
    # no more synapses than the paper's 64x64 torus has and half as many again, no more synapse steps than
    # the runaway's; a batch counts as a third of its nets at this size
    many = max(1, nets // 3)
    while gy > 1 and gx * gy * npc * fanout * many > 1.2e9:
        gy //= 2
    neurons = gx * gy * npc
    synapses = neurons * fanout * many
    top = {"step": 1, "resume": 300, "request": 400, "window": 300, "batch": 60, "simulate": 1100}[kind]
    steps = 1 if kind == "step" else _log_int(rng, 10, max(10, min(top, int(4e10 / synapses))))
    c = _case(kind, gx, gy, npc, fanout, mix if gx * gy > 1 else "local", steps, nets=nets)
    spikes = neurons * steps * _rate(c) / 1000.0
    if kind == "simulate":
        c["fp64"] = rng.random() < 0.15
        c["raster"] = spikes < 2e6 and rng.random() < 0.5
        c["weights"] = synapses < 2e7 and rng.random() < 0.5
    elif kind in ("request", "window", "resume"):
        c["raster"] = True
        if spikes > 2e6:
            c["steps"] = max(10, int(steps * 2e6 / spikes))
        c["weights"] = kind == "resume"
    return c


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def _config(case, seed):
    return workloads.custom(grid_x=case["gx"], grid_y=case["gy"], neurons_per_col=case["npc"],
                            exc_per_col=case["npc"] * 4 // 5, fanout=case["fanout"], pct_ring=MIX[case["mix"]],
                            seed=1 + int(seed), flags=eng.snn.FP64 if case["fp64"] else 0)


def _capacity(case):
    return case["gx"] * case["gy"] * case["npc"] * case["steps"] if case["raster"] else 0


def _drive(case, seed, steps):
    """Host events like the thalamic drive: one random neuron per column and millisecond gets 20 mV."""
    columns = case["gx"] * case["gy"]
    rng = np.random.default_rng(seed)
    ev = np.zeros(steps * columns, eng.snn.STIM_DTYPE)
    ev["t"] = np.repeat(np.arange(steps), columns)
    ev["gid"] = np.tile(np.arange(columns) * case["npc"], steps) + rng.integers(0, case["npc"], steps * columns)
    ev["q16"] = 20 * workloads.Q16
    return ev


def _connectome(case, seed):
    """Uneven rows around `fanout` synapses (the same lengths for every seed), to any neuron, excitatory delays
    of 1..20 ms, inhibitory of 1..3."""
    n = case["gx"] * case["gy"] * case["npc"]
    exc = np.arange(n) % case["npc"] < case["npc"] * 4 // 5
    rows = np.random.default_rng(n).integers(case["fanout"] * 6 // 10, case["fanout"] * 14 // 10 + 1, n)
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(rows)])
    src_exc = np.repeat(exc, rows)
    total = int(off[-1])
    return dict(row_off=off, tgt=rng.integers(0, n, total),
                delay=np.where(src_exc, rng.integers(1, 21, total), rng.integers(1, 4, total)),
                w=np.where(src_exc, 6 * workloads.Q16, -5 * workloads.Q16))


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if case["raster"]:
        # the caller's own spike buffers, four times what such a net emits; -1 behind the spikes
        n = case["gx"] * case["gy"] * case["npc"] * case["steps"]
        room = min(n, 1000 + int(4 * n * _rate(case) / 1000.0))
        s["t_buf"], s["gid_buf"], s["kept"] = np.full(room, -1, np.int32), np.full(room, -1, np.int32), 0
    if kind == "request":
        s["cfg"] = _config(case, seed)
    elif kind == "batch":
        nets = workloads.batch_workloads(case["nets"], first_seed=1000 + int(seed), side=(1, case["gx"]),
                                         fanouts=(100, min(400, case["fanout"]), case["fanout"]))
        s["nets"] = [eng.Network(c, raster_capacity=0) for c in nets]
        s["batch"] = eng.Batch(s["nets"])
    elif kind == "resume":
        cfg = _config(case, seed)
        s["net"] = eng.Network(cfg, raster_capacity=max(_capacity(case), 200 * case["gx"] * case["gy"] * case["npc"]),
                               explicit=_connectome(case, seed))
        s["net"].run(150)
        s["from"] = 150
        s["checkpoint"] = s["net"].save_state()
    else:
        s["net"] = eng.Network(_config(case, seed), raster_capacity=_capacity(case))
        if kind in ("step", "window"):
            s["net"].set_thalamic(False)
        if kind == "step":
            s["t"] = 0
            s["events"] = np.split(_drive(case, seed, 64), 64)
        if kind == "window":
            s["events"] = _drive(case, seed, case["steps"])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _counters(net):
    c = net.counters()
    return np.array([c[k] for k in ("t", "spikes", "e_all", "e_exc", "l_exc")], np.int64)


def _raster(s, t, gid):
    n = min(len(t), len(s["t_buf"]))
    for name, x in (("t_buf", t), ("gid_buf", gid)):
        s[name][:n] = x[:n]
        s[name][n:s["kept"]] = -1
    s["kept"] = n
    return {"spikes": len(t), "t": s["t_buf"], "gid": s["gid_buf"]}


def run(s):
    case = s["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "step":
        ev = s["events"][s["t"] % len(s["events"])]
        ev["t"] = s["t"]
        spikes = s["net"].run_host_counts(1, ev)
        s["t"] += 1
        return {"spikes": spikes, **s["net"].neurons()}
    if kind == "request":
        with eng.Network(s["cfg"], raster_capacity=_capacity(case)) as net:
            net.run(steps)
            return {**_raster(s, *net.raster()), "counters": _counters(net)}
    if kind == "batch":
        for net in s["nets"]:
            net.reset()
        s["batch"].run(steps)
        states = [net.neurons() for net in s["nets"]]
        return {"v": np.concatenate([x["v"] for x in states]), "u": np.concatenate([x["u"] for x in states]),
                "counters": np.stack([_counters(net) for net in s["nets"]])}
    net = s["net"]
    out = {}
    if kind == "window":
        net.reset()
        return _raster(s, *net.run_host(steps, s["events"], cap=len(s["t_buf"])))
    if kind == "resume":
        net.load_state(s["checkpoint"])
        net.run(steps)
        out.update(_raster(s, *net.raster(s["from"], s["from"] + steps)))
    else:
        net.reset()
        net.run(steps)
        if case["raster"]:
            out.update(_raster(s, *net.raster()))
    if case["weights"]:
        out["w"], out["sd"] = net.weights()
    out.update(net.neurons_f64() if case["fp64"] else net.neurons())
    out["counters"] = _counters(net)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _rate(case):
    """Mean rate (Hz) of such a net over a pass, as measured on this engine to about a factor of two."""
    m, steps = case["fanout"], case["steps"]
    if m < 120:
        return 6.0
    if m < 250:
        return 20.0
    if m < 320:
        return 75.0
    return 18.0 if steps <= 25 else 18.0 + 950.0 * (1.0 - 25.0 / steps)


def _one(neurons, fanout, steps, rate):
    """Bytes and operations of `steps` ms of one net: per synaptic event its target and weight (no more than
    every synapse once a step), every plastic derivative and neuron state in and out; 24 operations per
    neuron and step and one per event."""
    synapses = neurons * fanout
    events = synapses * min(1.0, rate / 1000.0) * steps
    moved = 6 * events + 0.8 * 8 * synapses + 24 * neurons * steps
    moved += (steps // 1000) * 0.8 * 8 * synapses
    return moved, 24.0 * neurons * steps + events


def work(case):
    neurons, steps, rate = case["gx"] * case["gy"] * case["npc"], case["steps"], _rate(case)
    if case["kind"] == "batch":
        parts = []
        for c in workloads.batch_workloads(case["nets"], side=(1, case["gx"]),
                                           fanouts=(100, min(400, case["fanout"]), case["fanout"])):
            parts.append(_one(workloads.n_neurons(c), c["fanout"], steps, _rate(dict(case, fanout=c["fanout"]))))
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if case["kind"] == "step":
        return {"bytes": 24 * neurons + 12 * case["gx"] * case["gy"], "flops": 24.0 * neurons}
    b, f = _one(neurons, case["fanout"], steps, rate)
    if case["kind"] == "request":
        b += 14 * neurons * case["fanout"]          # targets, weights, derivatives, incoming lists
    if case["raster"]:
        b += 8 * neurons * steps * rate / 1000.0
    if case["weights"]:
        b += 8 * neurons * case["fanout"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain numpy
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on arrays of counters; the first two words."""
    u = np.uint64
    mask = u(0xFFFFFFFF)
    x = [np.asarray(v, np.uint64) for v in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = x[0] * u(0xD2511F53), x[2] * u(0xCD9E8D57)
        x = [(p1 >> u(32)) ^ x[1] ^ u(k0), p1 & mask, (p0 >> u(32)) ^ x[3] ^ u(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x[0], x[1]


def _below(r, n):
    return ((r * np.uint64(n)) >> np.uint64(32)).astype(np.int64)


def _update(v, u, iq, exc):
    cur = iq * 2.0 ** -16
    for _ in range(2):
        v = v + 0.5 * (((0.04 * v + 5.0) * v + 140.0) - u + cur)
    u = u + np.where(exc, 0.02, 0.1) * (0.2 * v - u)
    fired = v >= 30.0
    return np.where(fired, -65.0, v), np.where(fired, u + np.where(exc, 8.0, 2.0), u), fired


def exact(case, seed):
    """Membrane state in 64 bits: of a closed-loop step, and of a one-column net in the double-precision mode
    within its first plasticity period.  None elsewhere: a float32 network's trajectory leaves the 64-bit one
    at the first threshold crossing that rounds the other way, and larger nets take too long."""
    npc, ne = case["npc"], case["npc"] * 4 // 5
    n = case["gx"] * case["gy"] * npc
    exc = np.arange(n) % npc < ne
    v, u = np.full(n, -65.0), np.full(n, 0.2 * -65.0)
    if case["kind"] == "step":
        ev = _drive(case, seed, 64)[: case["gx"] * case["gy"]]
        iq = np.zeros(n, np.int64)
        np.add.at(iq, ev["gid"], ev["q16"])
        v, u, _ = _update(v, u, iq, exc)
        return {"spikes": None, "v": v, "u": u}
    if not (case["kind"] == "simulate" and case["fp64"] and n == npc and case["steps"] <= 1000
            and n * case["fanout"] <= 400000):
        return None
    m, s = case["fanout"], 1 + int(seed)
    src, j = np.repeat(np.arange(n), m), np.tile(np.arange(m), n)
    r0, r1 = _philox(src, j, np.zeros_like(src), np.zeros_like(src), s)
    local = _below(r0, npc - 1)
    local += local >= src
    src_exc = exc[src]
    tgt = np.where(src_exc, local, _below(r0, ne)).reshape(n, m)
    delay = np.where(src_exc, 1 + _below(r1, 20), 1).reshape(n, m)
    weight = np.where(exc, 6, -5) * workloads.Q16
    due = np.zeros((21, n), np.int64)               # current arriving at step t in row t % 21
    for t in range(case["steps"]):
        iq, due[t % 21] = due[t % 21].copy(), 0
        th, _ = _philox(np.array([t]), np.array([0]), np.array([1]), np.array([0]), s)
        iq[_below(th, npc)] += 20 * workloads.Q16
        v, u, fired = _update(v, u, iq, exc)
        for p in np.flatnonzero(fired):
            np.add.at(due, ((t + delay[p]) % 21, tgt[p]), weight[p])
    out = {"spikes": None, "t": None, "gid": None} if case["raster"] else {}
    if case["weights"]:
        out.update(w=None, sd=None)
    return {**out, "v": v, "u": u, "counters": None}
