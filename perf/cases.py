"""The simulator's work, case by case, through its public entry points.

Two kinds of call carry it:

* ``steps``: ``Network.step(steps)`` and then ``Network.read_spikes()``, the loop of every
  simulation.  A pass returns its spikes (in arrays of the case's size, filled up with -1)
  and the dynamic state: U, I, R and the delay ring.
* ``deliver``: ``Network.deliver_spikes()``, phase 2 alone for a list of senders.  A pass
  returns the ring.

``n`` and ``k`` are the neuron and in-degree scales in permille of the Potjans-Diesmann
microcircuit; ``circuits`` > 0 makes a batch of that many uneven circuits with scales
drawn from 100 to n and 100 to k, run in groups of ``groups`` circuits.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_02019_gb300 as snn
import workload

_ENGINES = {"default": snn.ENGINE_DEFAULT, "graph": snn.ENGINE_GRAPH, "pipelined": snn.ENGINE_PIPELINED,
            "persistent": snn.ENGINE_PERSISTENT, "resident": snn.ENGINE_RESIDENT}
_RECORDS = {"plain": (snn.RECORD_PLAIN9, 9), "int8": (snn.RECORD_PACKED_I8, 5), "bf16": (snn.RECORD_PACKED_BF16, 6),
            "blocked6": (snn.RECORD_BLOCKED6, 6), "blocked4": (snn.RECORD_BLOCKED4, 4),
            "blocked8": (snn.RECORD_BLOCKED8, 8)}


def _steps(name, n, k, steps, engine="default", record="plain", circuits=0, groups=0):
    return {"name": name, "kind": "steps", "n": n, "k": k, "steps": steps, "engine": engine, "record": record,
            "circuits": circuits, "groups": groups}


def _deliver(name, n, k, senders, order="random", engine="default", record="plain"):
    return {"name": name, "kind": "deliver", "n": n, "k": k, "senders": senders, "order": order, "engine": engine,
            "record": record}


def listed():
    return [
        # a closed loop around the tiny circuit: 1 ms of biological time, then its spikes
        _steps("loop_1ms", 100, 100, 10),
        # the tiny circuit's whole run: 1,000 steps at 0.1x neurons and in-degrees
        _steps("tiny_1000", 100, 100, 1000),
        # the full microcircuit on the default engine, 1 s of biological time in one call
        _steps("full_1s", 1000, 1000, 10000),
        # the full microcircuit on the resident engine, one launch per 1,024-step call
        _steps("full_resident", 1000, 1000, 1024, engine="resident"),
        # the precision form (int8 weights) of a circuit of odd size, 0.2 s
        _steps("int8_200ms", 437, 1000, 2000, record="int8"),
        # a parameter sweep: 16 uneven circuits in one batch, 8 at a time, 0.1 s
        _steps("batch16", 400, 400, 1000, circuits=16, groups=8),
        # the scaled-up circuit (4x neurons) at reduced in-degrees, bfloat16 weights, 50 ms
        _steps("x4_bf16", 4000, 200, 500, record="bf16"),
        # target-blocked records in the step loop (two kernels per step), 50 ms
        _steps("blocked8_loop", 500, 1000, 500, record="blocked8"),
        # phase 2 alone under heavy load, a synchronous burst: plain rows ...
        _deliver("deliver_plain", 500, 1000, 8192),
        # ... exact target-blocked rows at full scale, the largest burst ...
        _deliver("deliver_blocked8", 1000, 1000, 20480, record="blocked8"),
        # ... target-blocked rows with bfloat16 weights, a smaller burst ...
        _deliver("deliver_blocked4", 500, 1000, 2048, record="blocked4"),
        # ... and the resident engine's block-major rows, senders in index order
        _deliver("deliver_resident", 500, 1000, 8192, order="sorted", engine="resident"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    deliver = rng.random() < 0.4
    form = rng.choice(["plain", "plain", "int8", "bf16", "resident", "resident", "blocked4", "blocked6", "blocked8"])
    engine, record = ("resident", "plain") if form == "resident" else ("default", form)
    n = _log_int(rng, 30, 1000 if engine == "resident" or record.startswith("blocked") else 4000)
    k = _log_int(rng, 100, max(101, min(1000, 500000 // n)))
    if deliver:
        case = _deliver("", n, k, _log_int(rng, 1, 20480), rng.choice(["random", "sorted"]), engine, record)
    else:
        if engine == "default" and not record.startswith("blocked"):
            engine = rng.choice(["default", "default", "default", "graph", "persistent"])
        circuits = rng.choice([0, 0, rng.randint(2, 12)]) if engine == "default" and record == "plain" else 0
        if circuits:
            n, k = rng.randint(150, 500), rng.randint(150, 500)
        groups = rng.randint(0, circuits) if circuits else 0
        case = _steps("", n, k, _log_int(rng, 1, 2500), engine, record, circuits, groups)
    del case["name"]
    return case


def _scales(case):
    """(neuron scale, in-degree scale) of every circuit of a case."""
    if not case.get("circuits"):
        return [(case["n"], case["k"])]
    rng = np.random.Generator(np.random.Philox(2026))
    return [(int(rng.integers(100, case["n"] + 1)), int(rng.integers(100, case["k"] + 1)))
            for _ in range(case["circuits"])]


def prepare(case, seed):
    model = workload.microcircuit_model()
    net_seed = 1 + seed % (1 << 40)
    record = _RECORDS[case["record"]][0]
    engine = _ENGINES[case["engine"]]
    if case.get("circuits"):
        circuits = [(n, k, net_seed * 4096 + c) for c, (n, k) in enumerate(_scales(case))]
        net = snn.Network(model, circuits=circuits, engine=engine, record_format=record)
        if case["groups"]:
            net.set_circuit_groups(case["groups"])
    else:
        net = snn.Network(model, case["n"], case["k"], seed=net_seed, engine=engine, record_format=record)
    state = {"case": case, "net": net, "t": 0, "views": {}}
    if case["kind"] == "deliver":
        rng = np.random.default_rng(seed)
        spikers = rng.integers(0, net.n_neurons, case["senders"], dtype=np.int32)
        if case["order"] == "sorted":
            spikers.sort()
        state["spikers"] = torch.from_numpy(spikers).to(net.device)
        state["t_spike"] = int(rng.integers(0, 10000))
        npad = int(net.layout().n_neurons_padded)
        state["views"] = {"ring": net.device_view("ring", torch.int32, 64 * npad)}
    else:
        room = 200 + int(1.5 * sum(_spikes(n, k, case["steps"]) for n, k in _scales(case)))
        state["steps"], state["neurons"] = np.full(room, -1, np.int64), np.full(room, -1, np.int32)
    return state


def run(state):
    case, net = state["case"], state["net"]
    if case["kind"] == "deliver":
        net.deliver_spikes(state["spikers"], state["t_spike"])
        return state["views"]
    net.step(case["steps"])
    steps, neurons = net.read_spikes()
    state["steps"][len(steps):] = -1
    state["neurons"][len(steps):] = -1
    state["steps"][: len(steps)] = steps
    state["neurons"][: len(steps)] = neurons
    state["t"] += case["steps"]
    views = state["views"].get(state["t"] & 1)  # the buffers that hold U and R alternate
    if views is None:
        n, npad = net.n_neurons, int(net.layout().n_neurons_padded)
        views = {"U": net.device_view("U", torch.float32, n), "I": net.device_view("I", torch.float32, n),
                 "R": net.device_view("R", torch.uint8, n), "ring": net.device_view("ring", torch.int32, 64 * npad)}
        state["views"][state["t"] & 1] = views
    return {"steps": state["steps"], "neurons": state["neurons"], **views}


def _sizes(model, n, k):
    """Population sizes and the pair counts [target][source] of one circuit."""
    nb = [(m * n + 500) // 1000 for m in model.n_full]
    pairs = [[int(math.floor(model.conn_p[b][a] * (model.n_full[a] * k / 1000.0) * nb[b] + 0.5)) for a in range(8)]
             for b in range(8)]
    return nb, pairs


def _spikes(n, k, steps):
    """Spikes of a run at the circuit's mean rate: 3.75e-4 per neuron and step at full
    in-degrees and about 1 / k^0.92 of that at others."""
    return 3.75e-4 * (k / 1000.0) ** -0.92 * 77.169 * n * steps


def work(case):
    """Bytes: every neuron's U, I, R once in and out and its ring entries of the steps read
    and cleared; every synaptic event's record once and every spike once out.  Phase 2
    alone: records, senders with their row bounds, and the ring entries that receive input
    read and written."""
    model = workload.microcircuit_model()
    rec = _RECORDS[case["record"]][1]
    nbytes = flops = 0.0
    for n, k in _scales(case):
        nb, pairs = _sizes(model, n, k)
        neurons, synapses = sum(nb), sum(map(sum, pairs))
        if case["kind"] == "deliver":
            events = case["senders"] * synapses / neurons
            entries = 28.0 * neurons * (1.0 - math.exp(-events / (28.0 * neurons)))
            nbytes += events * rec + case["senders"] * 20 + 8 * entries
            flops += events
        else:
            spikes = _spikes(n, k, case["steps"])
            events = spikes * 0.95 * synapses / neurons
            nbytes += neurons * (18 + 8 * min(64, case["steps"])) + events * rec + 8 * spikes
            flops += 9.0 * neurons * case["steps"] + events
    return {"bytes": nbytes, "flops": flops}


# ---- the same steps in 64 bits, from numpy alone -------------------------------------

def _philox(seed, tag, counter, blocks):
    """`blocks` consecutive Philox4x64-10 outputs from the 256-bit counter on: [blocks][4]."""
    g = np.random.Philox(key=seed | (tag << 64), counter=(counter - 1) % (1 << 256))
    return g.random_raw(4 * blocks).reshape(blocks, 4)


def _below(x, n):
    """floor(x n / 2^64) for 64-bit x and n below 2^32."""
    lo = (x & np.uint64(0xFFFFFFFF)) * np.uint64(n)
    return (((x >> np.uint64(32)) * np.uint64(n) + (lo >> np.uint64(32))) >> np.uint64(32)).astype(np.int64)


def _gauss(u, v):
    """The two Box-Muller normals of two 64-bit words."""
    f = lambda x: ((x >> np.uint64(11)).astype(np.float64) + 0.5) / 2.0 ** 53  # noqa: E731
    r, th = np.sqrt(-2.0 * np.log(f(u))), 2.0 * math.pi * f(v)
    return r * np.cos(th), r * np.sin(th)


def _bf16(w_fx):
    pa = torch.from_numpy(w_fx.astype(np.float32) / np.float32(4096.0))
    return np.rint(pa.to(torch.bfloat16).to(torch.float64).numpy() * 4096.0).astype(np.int64)


def _int8(w_fx):
    lo, hi = int(w_fx.min()), int(w_fx.max())
    base, step = lo + (hi - lo) // 2, max(1, -((lo - hi) // 254))
    x = (w_fx - base) / step
    code = np.clip(np.sign(x) * np.floor(np.abs(x) + 0.5), -127, 127).astype(np.int64)
    return base + code * step


def exact(case, seed):
    """U and I after the first pass with the neuron state in 64 bits (the synaptic input is
    an integer either way).  Only for runs short enough that no spike falls on another step
    in 32 bits, on circuits that numpy draws in a few seconds; a delivered ring is integer."""
    if case["kind"] == "deliver" or case.get("circuits") or case["steps"] > 32:
        return None
    m = workload.microcircuit_model()
    nb, pairs = _sizes(m, case["n"], case["k"])
    if sum(map(sum, pairs)) > 10_000_000:
        return None
    net_seed = 1 + seed % (1 << 40)
    off = np.concatenate([[0], np.cumsum(nb)])
    n, steps = int(off[-1]), case["steps"]
    ts, tm = m.tau_syn_ms, m.tau_m_ms
    w_f = m.C_m_pF * (ts - tm) / (ts * tm * ((tm / ts) ** (tm / (ts - tm)) - (tm / ts) ** (ts / (ts - tm))))
    p11, p22 = math.exp(-m.dt_ms / ts), math.exp(-m.dt_ms / tm)
    beta = ts * tm / (tm - ts)
    p21 = p11 * beta / m.C_m_pF * (math.exp(m.dt_ms / beta) - 1.0)
    theta, reset = m.u_thr_mV - m.u_rest_mV, m.u_reset_mV - m.u_rest_mV
    t_ref = int(round(m.tau_ref_ms / m.dt_ms))
    w_ext = int(round(w_f * m.w_ext_mV * 4096.0))

    # the network: synapse k of pair (a, b) from counter (k, a, b, 0)
    pre, post, weight, delay = [], [], [], []
    for a in range(8):
        for b in range(8):
            count = pairs[b][a]
            if count == 0:
                continue
            r = _philox(net_seed, 0xC0, (a << 64) | (b << 128), count)
            pre.append(off[a] + _below(r[:, 0], nb[a]))
            post.append(off[b] + _below(r[:, 1], nb[b]))
            zc, zs = _gauss(r[:, 2], r[:, 3])
            mu, sd = next(((x, y) for s, t, x, y in m.overrides if (s, t) == (a, b)), (m.w_mean_mV[a], m.w_sd_mV[a]))
            amp = mu + sd * zc
            x = (np.maximum(amp, 0.0) if mu >= 0 else np.minimum(amp, 0.0)) * w_f * 4096.0
            w = (np.sign(x) * np.floor(np.abs(x) + 0.5)).astype(np.int64)
            weight.append(_int8(w) if case["record"] == "int8" else
                          _bf16(w) if case["record"] in ("bf16", "blocked4") else w)
            delay.append(np.clip(np.floor((m.d_mean_ms[a] + m.d_sd_ms[a] * zs) / m.dt_ms + 0.5), 1, 63).astype(np.int64))
    pre, post, weight, delay = map(np.concatenate, (pre, post, weight, delay))
    order = np.argsort(pre, kind="stable")
    post, weight, delay = post[order], weight[order], delay[order]
    row = np.concatenate([[0], np.cumsum(np.bincount(pre, minlength=n))])

    # thalamic counts: word i mod 4 of counter (t, i div 4, 0, 0), by inversion of the CDF
    pop = np.repeat(np.arange(8), nb)
    words = np.stack([_philox(net_seed, 0x7A, q << 64, steps) for q in range((n + 3) // 4)], axis=1)
    words = (words.reshape(steps, -1)[:, :n] >> np.uint64(1)).astype(np.float64) / 2.0 ** 63
    count = np.zeros((steps, n), np.int64)
    lam = np.asarray(m.k_ext)[pop] * m.nu_th_hz * m.dt_ms * 1e-3
    cdf, pk = np.exp(-lam), np.exp(-lam)
    for j in range(1, 25):
        count += words >= cdf
        pk = pk * lam / j
        cdf = cdf + pk

    u0 = np.stack([_philox(net_seed, 0x1A, i, 1)[0] for i in range(n)])
    mean, sd = np.asarray(m.u0_mean_mV)[pop], np.asarray(m.u0_sd_mV)[pop]
    U = (mean + sd * _gauss(u0[:, 0], u0[:, 1])[0] - m.u_rest_mV).astype(np.float32).astype(np.float64)
    I, R = np.zeros(n), np.zeros(n, np.int64)
    W = np.zeros((64, n), np.int64)
    for t in range(steps):
        inp = (W[t % 64] + count[t] * w_ext) / 4096.0
        W[t % 64] = 0
        x = p22 * U + p21 * I
        free = R == 0
        spike = free & (x >= theta)
        U = np.where(free & ~spike, x, reset)
        R = np.where(spike, t_ref, np.maximum(R - 1, 0))
        I = p11 * I + inp
        for s in np.flatnonzero(spike):
            e = slice(row[s], row[s + 1])
            np.add.at(W, ((t + delay[e]) % 64, post[e]), weight[e])
    return {"steps": None, "neurons": None, "U": U, "I": I, "R": None, "ring": None}
