"""Performance cases: the work that users of this library have it do.

A case names a balanced random network (or an explicit edge list) by its
sizes and one way of using it through the public entry points of
``paper_2109_12855_gb300``:

* ``simulate``  the time-driven cycle of a built network (``snn_simulate``),
  then its state, ring buffer and spike raster; static, or with STDP on its
  E->E synapses (then also the plastic weights);
* ``step``      one interval through the single calls (``snn_update`` and
  ``snn_deliver_pending``), as a program that looks at every interval has it;
* ``deliver``   one caller's spike list into the ring buffer (``snn_deliver``);
* ``edges``     the same on a network given as an explicit edge list;
* ``build``     a network from its parameters to its first results (creation,
  connection, 10 ms of simulation, destruction);
* ``serve``     a batch of small requests through the server, submitted at
  once, to their spike trains;
* ``exchange``  one network held as target partitions with the device
  exchange (graph-replayed intervals).

Sizes come from the repository's workloads (balanced-1250, balanced-112500,
balanced-562500, the serving stream) or lie between them.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_2109_12855_gb300 import partition, snn

SLOTS = 32
DT = 1e-4                       # seconds per step
NU = 25757.293701171875         # drive of the 112,500-neuron benchmark (8 Hz)
PSP_MV, G = 0.1, 5.0
STDP_ALPHA, STDP_MU = 0.0513, 0.4


def _net(n, k, fmt, sd=0.0, d_lo=15, d_hi=15, nu=NU):
    """A balanced network with 4:1 E:I neurons and inputs."""
    n_i, k_i = n // 5, k // 5
    return dict(n_e=n - n_i, n_i=n_i, k_e=k - k_i, k_i=k_i, fmt=fmt, sd=sd,
                d_lo=d_lo, d_hi=d_hi, nu=nu)


def listed():
    return [
        # the paper's network at its smallest, active: intervals of ~50 spikes,
        # where launches and latency count
        dict(name="simulate 1250 fp32", kind="simulate", steps=2000, stdp=0,
             **_net(1250, 100, 0, d_lo=10, d_hi=20, nu=20000.0)),
        # a network of the serving stream's middle, odd size, run alone: BF16
        # records with spread weights and mixed delays, a short last interval
        dict(name="simulate 20003 bf16 spread", kind="simulate", steps=1005,
             stdp=0, **_net(20003, 2000, 1, 0.1, 10, 20)),
        # the headline benchmark: 1.27e9 synapses, FP32 records, 200 ms
        dict(name="simulate 112500 fp32", kind="simulate", steps=2000, stdp=0,
             **_net(112500, 11250, 0)),
        # the largest benchmark: 6.3e9 synapses, BF16, mixed delays, spread
        dict(name="simulate 562500 bf16 spread", kind="simulate", steps=500,
             stdp=0, **_net(562500, 11250, 1, 0.1, 10, 20)),
        # plastic E->E synapses on the 1.27e9-synapse network
        dict(name="simulate 112500 bf16 stdp", kind="simulate", steps=500,
             stdp=1, **_net(112500, 11250, 1)),
        # the smallest call: a few dozen spikes of a small network
        dict(name="deliver 1250 fp32", kind="deliver", hz=40.0, span=10,
             **_net(1250, 100, 0, d_lo=10, d_hi=20)),
        # one recorded interval of the 1.27e9-synapse network, replayed
        dict(name="deliver 112500 fp32", kind="deliver", hz=8.0, span=15,
             **_net(112500, 11250, 0)),
        # an explicit connectome: ragged rows (sources and targets drawn with
        # a heavy tail), all delays from 1 step up, own FP32 weights
        dict(name="edges 10007 fp32", kind="edges", n=10007, m=2000003, fmt=0,
             d_lo=1, d_hi=30, hz=30.0, span=1),
        # a program that looks at every interval: FP32 weights with spread
        dict(name="step 50021 fp32 spread", kind="step",
             **_net(50021, 1000, 0, 0.1, 10, 20)),
        # a user's whole session with a middle-sized network
        dict(name="build 30011 bf16 spread", kind="build", steps=100,
             **_net(30011, 3000, 1, 0.1, 10, 20)),
        # eight small requests of the serving stream, all at once
        dict(name="serve 8", kind="serve", requests=8, n_lo=1250, n_hi=20000,
             ms_lo=100.0, ms_hi=300.0),
        # the benchmark's partitioned arm at one GPU, BF16 records
        dict(name="exchange 112500 bf16", kind="exchange", parts=1, steps=1000,
             **_net(112500, 11250, 1)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate", "simulate", "simulate", "stdp", "deliver",
                       "deliver", "edges", "step", "build", "serve",
                       "exchange"])
    fmt = rng.choice([0, 1])
    sd = rng.choice([0.0, 0.1])
    d = rng.choice([(15, 15), (10, 20), (10, 20), (8, 23)])

    def net(lo, hi, fmt=fmt, sd=sd):
        n = _log_int(rng, lo, hi)
        k = max(5, min(n // 10, 11250))
        return _net(n, k, fmt, sd, *d)

    if kind == "simulate":
        return dict(kind="simulate", steps=rng.randrange(200, 2001), stdp=0,
                    **net(1250, 112500))
    if kind == "stdp":
        return dict(kind="simulate", steps=rng.randrange(100, 501), stdp=1,
                    **net(2000, 60000, sd=0.0))
    if kind == "deliver":
        return dict(kind="deliver", hz=round(math.exp(rng.uniform(0.0, 4.0)), 2),
                    span=rng.randrange(1, d[0] + 1), **net(1250, 112500))
    if kind == "edges":
        n = _log_int(rng, 300, 40000)
        return dict(kind="edges", n=n, m=_log_int(rng, 20 * n, 100 * n),
                    fmt=fmt, d_lo=rng.randrange(1, 11), d_hi=rng.randrange(11, 31),
                    hz=round(math.exp(rng.uniform(0.0, 4.0)), 2),
                    span=rng.randrange(1, 11))
    if kind == "step":
        return dict(kind="step", **net(1250, 100000))
    if kind == "build":
        return dict(kind="build", steps=rng.randrange(20, 201), **net(1250, 50000))
    if kind == "serve":
        return dict(kind="serve", requests=rng.randrange(2, 11), n_lo=1250,
                    n_hi=_log_int(rng, 2000, 20000), ms_lo=50.0,
                    ms_hi=float(rng.randrange(60, 301)))
    return dict(kind="exchange", parts=rng.randrange(1, 4),
                steps=rng.randrange(200, 1001), **net(2000, 112500))


# ---------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------
_stream = None


def _stream_of():
    """The one stream this program runs its networks and its reads on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _params(c, seed, **kw):
    p = snn.params(n_exc=c["n_e"], n_inh=c["n_i"], weight_format=c["fmt"],
                   seed=seed, nu_ext=c["nu"], n_slots=SLOTS, **kw)
    p.w_ext = snn.snn_psc_weight_for_psp(p, PSP_MV)
    return p


def _conn(c, p, seed):
    w = p.w_ext
    return snn.conn_params(k_exc=c["k_e"], k_inh=c["k_i"], w_exc=w,
                           w_inh=-G * w, sd_exc=c["sd"] * w,
                           sd_inh=c["sd"] * G * w, d_lo=c["d_lo"],
                           d_hi=c["d_hi"], seed=seed + 1000, clip_exc=1,
                           clip_inh=0)


def _log_cap(c, steps):
    """Room for the spikes of a pass at 150 Hz."""
    return int((c["n_e"] + c["n_i"]) * steps * DT * 150.0) + 8192


def _spikes(n, hz, span, seed):
    """Spike list of ``span`` steps: every neuron fires with probability
    hz dt in each step (at least one spike)."""
    g = np.random.Generator(np.random.PCG64(seed))
    hit = np.nonzero(g.random((span, n)) < hz * DT)
    t, src = (hit if len(hit[0]) else (np.zeros(1, int), np.zeros(1, int)))
    return src.astype(np.int32), t.astype(np.int32)


def _edge_list(c, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    n, m = c["n"], c["m"]
    src = np.minimum((n * g.random(m) ** 2).astype(np.uint32), n - 1)
    tgt = np.minimum((n * g.random(m) ** 1.5).astype(np.uint32), n - 1)
    d = g.integers(c["d_lo"], c["d_hi"] + 1, m).astype(np.uint8)
    w = g.normal(0.0, 25.0, m).astype(np.float32).astype(np.float64)
    if c["fmt"] == 1:      # weights a BF16 record holds as they are
        w = torch.from_numpy(w).to(torch.bfloat16).double().numpy()
    return src, tgt, d, w


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _out_buffers(n):
    f = dict(dtype=torch.float32, device="cuda")
    return dict(V=torch.empty(n, **f), I=torch.empty(n, **f),
                J=torch.empty(n, **f),
                refr=torch.empty(n, dtype=torch.int32, device="cuda"),
                rb=torch.empty((SLOTS, n), **f))


def _random_state(c, seed):
    """A state in the middle of a run: potentials below threshold, currents
    of a few dozen pA, some neurons refractory, input waiting in the ring."""
    n = c["n_e"] + c["n_i"]
    g = np.random.Generator(np.random.PCG64(seed + 7))
    V = g.uniform(0.0, 20.0, n).astype(np.float32)
    I = g.normal(50.0, 50.0, n).astype(np.float32)
    J = g.normal(0.0, 200.0, n).astype(np.float32)
    refr = np.where(g.random(n) < 0.1, g.integers(1, 21, n), 0).astype(np.int32)
    rb = g.normal(0.0, 40.0, (SLOTS, n)).astype(np.float32)
    return V, I, J, refr, rb


def prepare(case, seed):
    c, kind = case, case["kind"]
    stream = _stream_of()
    sp = stream.cuda_stream
    st = dict(case=c, seed=seed)
    if kind == "serve":
        fmt = 1
        st["server"] = _Server(8 << 30, fmt)
        st["requests"] = _requests(c, seed, fmt)
        return st
    if kind == "build":
        st.update(_out_buffers(c["n_e"] + c["n_i"]))
        return st
    with torch.cuda.stream(stream):
        if kind == "edges":
            p = snn.params(n_exc=c["n"], n_inh=0, weight_format=c["fmt"],
                           n_slots=SLOTS, seed=seed)
            net = snn.Net(p, sp)
            net.connect_edges(*_edge_list(c, seed))
            net.finalize()
            n = c["n"]
        elif kind == "exchange":
            p = _params(c, seed)
            conn = _conn(c, p, seed)
            n = p.n_exc + p.n_inh
            nets = [partition.create(p, conn, lo, hi, sp)
                    for lo, hi in partition.split(n, c["parts"])]
            partition.agree_bounds(nets)
            for x in nets:
                x.finalize()
            st["nets"] = nets
            st["exchange"] = partition.DeviceExchange(nets)
            st["out"] = [_out_buffers(x.n) for x in nets]
            stream.synchronize()
            return st
        else:
            cap = _log_cap(c, c["steps"]) if kind == "simulate" else 0
            p = _params(c, seed, spike_log_capacity=cap)
            net = snn.Net(p, sp)
            if c.get("stdp"):
                # the fixed point of the rule at the initial E weight; the
                # usual small learning rate, so that a run keeps its rate
                snn.snn_set_stdp(net.h, snn.stdp_params(
                    lam=0.01, alpha=STDP_ALPHA, mu=STDP_MU, w_max=100.0,
                    w0=p.w_ext * STDP_ALPHA ** (1.0 / (1.0 - STDP_MU))))
            net.connect_fixed_indegree(_conn(c, p, seed))
            net.finalize()
            n = net.n
            if kind == "simulate":
                st["src"] = torch.empty(cap, dtype=torch.int32, device="cuda")
                st["t"] = torch.empty(cap, dtype=torch.int32, device="cuda")
                st["raster"] = torch.empty(cap, dtype=torch.int64, device="cuda")
                if c["stdp"]:
                    st["w"] = torch.empty(net.stats().n_synapses,
                                          dtype=torch.float32, device="cuda")
            if kind == "step":
                V, I, J, refr, rb = _random_state(c, seed)
                net.write_state(V, I, J, refr)
                snn.snn_write_rb(net.h, rb)
                st["interval"] = net.stats().interval
        if kind in ("deliver", "edges"):
            src, t = _spikes(n, c["hz"], c["span"], seed + 11)
            st["src"], st["t"] = _dev(src), _dev(t)
        st["net"] = net
        st.update(_out_buffers(n))
    stream.synchronize()
    return st


class _Server:
    """A server handle that is given back with its state."""

    def __init__(self, budget, fmt):
        self.h = snn.snn_server_create(budget, fmt)

    def __del__(self):
        snn.snn_server_destroy(self.h)


def _requests(c, seed, fmt):
    """Small networks of the serving stream: log-uniform sizes, K = N/10,
    BF16 records with spread weights, mixed delays; the sizes are the case's,
    each network's own seed comes from the state's."""
    g = np.random.Generator(np.random.PCG64(c["n_hi"] + c["requests"]))
    out = []
    for i in range(c["requests"]):
        n = int(round(math.exp(g.uniform(math.log(c["n_lo"]),
                                         math.log(c["n_hi"])))))
        net = _net(n, max(5, n // 10), fmt, 0.1, 10, 20)
        p = _params(net, seed + i)
        steps = int(round(g.uniform(c["ms_lo"], c["ms_hi"]) * 10))
        out.append(snn.request(p, _conn(net, p, seed + i), steps, user_tag=i,
                               record_spikes=True))
    return out


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _read_state(st, net, out=None):
    o = st if out is None else out
    snn.snn_read_state(net.h, o["V"], o["I"], o["J"], o["refr"])
    snn.snn_read_rb(net.h, o["rb"])
    return {k: o[k] for k in ("V", "I", "J", "refr", "rb")}


def run(state):
    st, c, kind = state, state["case"], state["case"]["kind"]
    with torch.cuda.stream(_stream_of()):
        if kind == "simulate":
            net = st["net"]
            snn.snn_simulate(net.h, c["steps"])
            out = _read_state(st, net)
            # the raster of this pass, by time and neuron
            k = min(snn.snn_read_spikes(net.h, st["src"], st["t"]), len(st["src"]))
            key = (st["t"][:k].long() << 24) | st["src"][:k].long()
            st["raster"].fill_(-1)
            st["raster"][:k] = torch.sort(key).values
            out["raster"] = st["raster"]
            if c["stdp"]:
                snn.snn_read_weights(net.h, st["w"])
                out["w"] = st["w"]
            return out
        if kind == "step":
            net = st["net"]
            snn.snn_update(net.h, snn.SNN_T_DEVICE, st["interval"])
            snn.snn_deliver_pending(net.h)
            return _read_state(st, net)
        if kind in ("deliver", "edges"):
            net = st["net"]
            snn.snn_deliver(net.h, st["src"], st["t"], want_events=False)
            snn.snn_read_rb(net.h, st["rb"])
            return st["rb"]
        if kind == "build":
            p = _params(c, st["seed"])
            with snn.Net(p, _stream_of().cuda_stream) as net:
                net.connect_fixed_indegree(_conn(c, p, st["seed"]))
                net.finalize()
                snn.snn_simulate(net.h, c["steps"])
                out = _read_state(st, net)
                out["spikes"] = snn.snn_read_spike_stats(net.h, net.n)[0]
            return out
        if kind == "exchange":
            partition.simulate_exchanged(st["nets"], st["exchange"], c["steps"],
                                         graph_intervals=8)
            return [_read_state(st, x, o) for x, o in zip(st["nets"], st["out"])]
    # serve
    sv = st["server"].h
    ids = [snn.snn_server_submit(sv, r) for r in st["requests"]]
    left, last = list(ids), -1
    while left:
        active = snn.snn_server_step(sv)
        left = [i for i in left
                if snn.snn_server_poll(sv, i).state in (0, 1, 2)]
        steps = snn.snn_server_get_stats(sv).steps
        if left and active == 0:
            time.sleep(1e-4)            # nothing on the GPU yet
        elif left and steps == last:
            time.sleep(2e-5)            # every lane busy
        last = steps
    out = []
    for i, req in zip(ids, st["requests"]):
        r = snn.snn_server_poll(sv, i)
        src, t = snn.snn_server_spikes(sv, i)
        # the raster by time and neuron, in room for 150 Hz
        raster = np.full(int(r.n_neurons * req.n_steps * DT * 150.0) + 8192, -1)
        k = min(len(src), len(raster))
        raster[:k] = np.sort((t.astype(np.int64) << 24) | src)[:k]
        out.append([raster, r.state, r.events])
        snn.snn_server_release(sv, i)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _rate(c):
    """About the rate of these networks under the drive (Hz), from a few
    measured ones: 46 at in-degree 100, 39 at 1,125, 8 at 11,250."""
    k = c["k_e"] + c["k_i"]
    x = math.log10(max(k, 100))
    return 46.0 - 7.0 * min(x - 2.0, 1.05) / 1.05 - 31.0 * max(0.0, x - 3.05)


def _event_bytes(c):
    """A synapse at its least: a 16-bit place in the window of its target's
    group, and its weight as held (none of its own where all are equal)."""
    w = 0 if c.get("sd", 1.0) == 0.0 else (4 if c["fmt"] == 0 else 2)
    return 2 + w


def _net_work(c, steps, hz, updated=True):
    n, k = c["n_e"] + c["n_i"], c["k_e"] + c["k_i"]
    spikes = n * hz * DT * steps
    events = spikes * k
    b = events * _event_bytes(c) + spikes * 16 + n * SLOTS * 4
    if c.get("stdp"):
        b += events * 0.64 * 8
    if updated:
        b += n * 32
    # one addition an event, about a dozen operations a neuron and step
    return dict(bytes=b, flops=events + (12.0 * n * steps if updated else 0.0))


def work(case):
    c, kind = case, case["kind"]
    if kind in ("simulate", "exchange"):
        return _net_work(c, c["steps"], _rate(c))
    if kind == "step":
        return _net_work(c, c["d_lo"], 30.0)
    if kind == "deliver":
        return _net_work(c, c["span"], c["hz"], updated=False)
    if kind == "edges":
        events = max(1.0, c["n"] * c["hz"] * DT * c["span"]) * c["m"] / c["n"]
        return dict(bytes=events * _event_bytes(c) + c["n"] * SLOTS * 4.0,
                    flops=events)
    if kind == "build":
        w = _net_work(c, c["steps"], _rate(c))
        syn = (c["n_e"] + c["n_i"]) * (c["k_e"] + c["k_i"])
        # every synapse written once; a draw of ten rounds for each
        return dict(bytes=w["bytes"] + syn * _event_bytes(c),
                    flops=w["flops"] + syn * 40.0)
    b = f = 0.0
    n = math.sqrt(c["n_lo"] * c["n_hi"])
    for _ in range(c["requests"]):
        x = _net(int(n), max(5, int(n) // 10), 1, 0.1, 10, 20)
        w = _net_work(x, 5.0 * (c["ms_lo"] + c["ms_hi"]), _rate(x))
        syn = n * n / 10
        b += w["bytes"] + syn * 4
        f += w["flops"] + syn * 40.0
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((b >> 32) & _M32) ^ c1 ^ k0, b & _M32,
                          ((a >> 32) & _M32) ^ c3 ^ k1, a & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _drawn_synapses(c, seed, w, count):
    """The fixed in-degree rule's synapses whose source has count > 0:
    (source, target, delay, weight) in blocks."""
    n, k = c["n_e"] + c["n_i"], c["k_e"] + c["k_i"]
    per = max(1, (1 << 25) // k)
    kk = torch.arange(k, device="cuda")
    for lo in range(0, n, per):
        tgt = torch.arange(lo, min(n, lo + per), device="cuda")
        a = tgt[:, None].expand(-1, k).reshape(-1)
        b = kk[None, :].expand(len(tgt), -1).reshape(-1)
        z = torch.zeros_like(a)
        r0, r1, r2, r3 = _philox(a, b, z, z, seed + 1000)
        exc = b < c["k_e"]
        src = torch.where(exc, (r0 * c["n_e"]) >> 32,
                          c["n_e"] + ((r0 * c["n_i"]) >> 32))
        sel = torch.nonzero(count[src] > 0).flatten()
        exc = exc[sel]
        x = torch.where(exc, w, -G * w).double()
        if c["sd"]:
            u1 = (r2[sel].double() + 1.0) * 2.0 ** -32
            u2 = r3[sel].double() * 2.0 ** -32
            x = x + torch.where(exc, c["sd"] * w, c["sd"] * G * w) * (
                torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2))
            x = torch.where(exc, x.clamp(min=0.0), x)
        if c["fmt"] == 1:
            x = x.to(torch.bfloat16).double()
        d = c["d_lo"] + ((r1[sel] * (c["d_hi"] - c["d_lo"] + 1)) >> 32)
        yield src[sel], a[sel], d, x


def _add_spikes(rb, n, src, t, synapses):
    """rb[(t + d) mod S][target] += w over the synapses of every spike."""
    order = torch.argsort(src)
    s, tt = src[order], t[order]
    count = torch.bincount(s, minlength=n)
    first = torch.cumsum(count, 0) - count
    flat = rb.view(-1)
    for ss, tg, d, w in synapses(count):
        rep = count[ss]
        e = torch.repeat_interleave(torch.arange(len(ss), device="cuda"), rep)
        pos = torch.arange(len(e), device="cuda") - (
            torch.cumsum(rep, 0) - rep)[e] + first[ss[e]]
        cell = ((tt[pos] + d[e]) % SLOTS) * rb.shape[1] + tg[e]
        flat.index_add_(0, cell, w[e])


def _psc_weight():
    return snn.snn_psc_weight_for_psp(snn.params(), PSP_MV)


def _exact_step(c, seed):
    """One interval of iaf_psc_alpha neurons with exact integration, then the
    delivery of its spikes."""
    n, w, h = c["n_e"] + c["n_i"], _psc_weight(), 0.1
    D = c["d_lo"]
    V, I, J, refr, rb = (torch.from_numpy(a).cuda() for a in _random_state(c, seed))
    V, I, J, rb = V.double(), I.double(), J.double(), rb.double()
    refr = refr.long()
    a, b = 1.0 / 0.5, 1.0 / 10.0
    E = torch.linalg.matrix_exp(torch.tensor(
        [[-a * h, 0, 0], [h, -a * h, 0], [0, h / 250.0, -b * h]],
        dtype=torch.float64))
    lam = c["nu"] * h * 1e-3
    thr, p, F, k = [], math.exp(-lam), math.exp(-lam), 0
    while math.floor(F * 2.0 ** 32) < 2 ** 32 - 1:
        thr.append(math.floor(F * 2.0 ** 32))
        k += 1
        p *= lam / k
        F += p
    thr = torch.tensor(thr, device="cuda")
    ids = torch.arange(n, device="cuda")
    z = torch.zeros_like(ids)
    src, t = [], []
    for step in range(D):
        word = _philox(ids, z + (step >> 2), z, z + 2, seed)[step & 3]
        drive = torch.searchsorted(thr, word, right=True).double() * w
        V = torch.where(refr == 0, E[2, 0].item() * J + E[2, 1].item() * I
                        + E[2, 2].item() * V, V)
        refr = (refr - 1).clamp(min=0)
        I = E[1, 0].item() * J + E[1, 1].item() * I
        J = E[0, 0].item() * J + (math.e / 0.5) * (rb[step] + drive)
        rb[step] = 0.0
        fired = torch.nonzero(V >= 20.0).flatten()
        V[fired], refr[fired] = 0.0, 20
        src.append(fired)
        t.append(torch.full_like(fired, step))
    _add_spikes(rb, n, torch.cat(src), torch.cat(t),
                lambda cnt: _drawn_synapses(c, seed, w, cnt))
    return dict(V=V, I=I, J=J, refr=None, rb=rb)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        return _exact_step(c, seed)
    if kind not in ("deliver", "edges"):
        return None          # spiking dynamics: no value of their own in 64 bits
    n = c["n"] if kind == "edges" else c["n_e"] + c["n_i"]
    src, t = _spikes(n, c["hz"], c["span"], seed + 11)
    src, t = _dev(src).long(), _dev(t).long()
    rb = torch.zeros((SLOTS, n), dtype=torch.float64, device="cuda")
    if kind == "edges":
        e = [_dev(x.astype(np.int64)) for x in _edge_list(c, seed)[:3]]
        e.append(_dev(_edge_list(c, seed)[3]))
        _add_spikes(rb, n, src, t, lambda cnt: [e])
    else:
        _add_spikes(rb, n, src, t, lambda cnt: _drawn_synapses(
            c, seed, _psc_weight(), cnt))
    return rb
