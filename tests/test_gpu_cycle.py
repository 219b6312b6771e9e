"""snn_simulate's one-launch cycle against the same intervals run through the
single calls (snn_update, snn_deliver_pending): state, ring buffer, spikes,
counters and spike statistics agree bit for bit, for every store layout and at
the edges of its shapes (one tile and many, tiles wider than a CTA's threads, a
last tile of one neuron, intervals around the 16-step and 4-step groups, a
short last interval, more intervals than one launch takes, input already in
the ring buffer, a clock that starts off the 4-step blocks)."""
import numpy as np
import pytest

from gpu_common import need_gpu, stream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _net(n, k, fmt, sd, d_lo, d_hi, **kw):
    from paper_2109_12855_gb300 import snn
    n_i, k_i = n // 5, k // 5
    p = snn.params(n_exc=n - n_i, n_inh=n_i, weight_format=fmt, seed=11,
                   nu_ext=kw.pop("nu", 26000.0), spike_log_capacity=1 << 18,
                   **kw)
    w = snn.snn_psc_weight_for_psp(p, 0.1)
    p.w_ext = w
    net = snn.Net(p, stream())
    net.connect_fixed_indegree(snn.conn_params(
        k_exc=k - k_i, k_inh=k_i, w_exc=w, w_inh=-5 * w, sd_exc=sd * w,
        sd_inh=5 * sd * w, d_lo=d_lo, d_hi=d_hi, seed=5))
    net.finalize()
    g = np.random.Generator(np.random.PCG64(3))
    net.write_state(g.uniform(0, 20, n), g.normal(50, 50, n),
                    g.normal(0, 200, n),
                    np.where(g.random(n) < 0.2, g.integers(1, 21, n), 0))
    snn.snn_write_rb(net.h, g.normal(0, 40, (p.n_slots, n)).astype(np.float32))
    snn.snn_set_time(net.h, 7)
    return net


def _result(net):
    src, t = net.read_spikes()
    order = np.lexsort((src, t))
    from paper_2109_12855_gb300 import snn
    st = net.stats()
    return ([*net.read_state(), net.read_rb(), src[order], t[order]] +
            list(snn.snn_read_spike_stats(net.h, net.n)),
            (st.t_now, st.spikes, st.events_delivered, st.error_flags))


CASES = [
    # n, k, fmt, sd, d_lo, d_hi, steps, options
    pytest.param(1250, 100, 0, 0.0, 10, 20, 405, {}, id="fp32-uniform"),
    pytest.param(1251, 100, 0, 0.1, 15, 15, 95, {}, id="fp32-spread"),
    pytest.param(641, 64, 1, 0.1, 17, 23, 120, {}, id="bf16-integer-17"),
    pytest.param(900, 90, 1, 0.0, 8, 9, 83, {}, id="bf16-uniform-8"),
    pytest.param(700, 70, 1, 0.1, 3, 30, 31, {"acc_words": 2}, id="bf16-two-word"),
    pytest.param(2500, 60, 0, 0.0, 5, 6, 600, {"tile_width": 1250}, id="wide-tiles"),
    pytest.param(513, 20, 1, 0.1, 1, 2, 601, {"tile_width": 512}, id="launches-of-1-step"),
    pytest.param(64, 10, 0, 0.0, 32, 32, 70, {}, id="one-tile-32"),
    pytest.param(1250, 100, 0, 0.0, 10, 20, 200, {"nu": 0.0}, id="no-drive"),
]


@pytest.mark.parametrize("n,k,fmt,sd,d_lo,d_hi,steps,kw", CASES)
def test_cycle_equals_single_calls(n, k, fmt, sd, d_lo, d_hi, steps, kw):
    from paper_2109_12855_gb300 import snn
    with _net(n, k, fmt, sd, d_lo, d_hi, **dict(kw)) as a, \
            _net(n, k, fmt, sd, d_lo, d_hi, **dict(kw)) as b:
        D = a.stats().interval
        before = a.stats().kernel_launches
        snn.snn_simulate(a.h, steps)
        left = steps
        while left > 0:
            snn.snn_update(b.h, snn.SNN_T_DEVICE, min(D, left))
            snn.snn_deliver_pending(b.h)
            left -= D
        if not snn.snn_checked():  # (which runs the separate kernels)
            assert a.stats().kernel_launches - before == -(-(-(-steps // D)) // 256)
        (xs, cs), (ys, ds) = _result(a), _result(b)
        assert cs == ds and cs[3] == 0
        assert cs[1] > 0 or kw.get("nu") == 0.0
        for x, y in zip(xs, ys):
            assert np.array_equal(x.view(np.uint32 if x.itemsize == 4 else np.uint64),
                                  y.view(np.uint32 if y.itemsize == 4 else np.uint64))


def test_log_overflow_is_flagged():
    from paper_2109_12855_gb300 import snn
    p = snn.params(n_exc=400, n_inh=100, nu_ext=40000.0, spike_log_capacity=10)
    p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
    with snn.Net(p, stream()) as net:
        net.connect_fixed_indegree(snn.conn_params(
            k_exc=40, k_inh=10, w_exc=p.w_ext, w_inh=-5 * p.w_ext, d_lo=10,
            d_hi=20, seed=5))
        net.finalize()
        snn.snn_simulate(net.h, 300)
        st = net.stats()
        assert st.error_flags == snn.SNN_ERRF_SPIKE_LOG and st.spikes > 10
        src, t = np.zeros(10, np.uint32), np.zeros(10, np.int32)
        assert snn.snn_read_spikes(net.h, src, t) == st.spikes


def test_two_nets_on_two_streams():
    """Launches of two nets that each want every SM, queued alternately on two
    streams: both finish, each with the result it has alone."""
    import torch
    from paper_2109_12855_gb300 import snn
    results = []
    for together in (False, True):
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        nets = []
        for seed, s in zip((1, 2), streams):
            p = snn.params(n_exc=16000, n_inh=4000, weight_format=1, seed=seed,
                           nu_ext=26000.0)
            p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
            net = snn.Net(p, s.cuda_stream)
            net.connect_fixed_indegree(snn.conn_params(
                k_exc=160, k_inh=40, w_exc=p.w_ext, w_inh=-5 * p.w_ext,
                sd_exc=2.0, sd_inh=10.0, d_lo=10, d_hi=20, seed=seed))
            net.finalize()
            nets.append(net)
        for _ in range(6):
            for net in nets:
                snn.snn_simulate(net.h, 205)
                if not together:
                    snn.snn_sync(net.h)
        results.append([x for net in nets for x in (*net.read_state(), net.read_rb())])
        assert all(net.stats().error_flags == 0 for net in nets)
        for net in nets:
            net.close()
    for x, y in zip(*results):
        assert np.array_equal(x, y)


def test_cycle_in_a_captured_graph():
    """A call captured by the caller replays from the device clock."""
    import torch
    from paper_2109_12855_gb300 import snn
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    nets = []
    for _ in range(2):
        p = snn.params(n_exc=1000, n_inh=250, seed=4, nu_ext=26000.0)
        p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
        net = snn.Net(p, s.cuda_stream)
        net.connect_fixed_indegree(snn.conn_params(
            k_exc=80, k_inh=20, w_exc=p.w_ext, w_inh=-5 * p.w_ext, d_lo=10,
            d_hi=20, seed=5))
        net.finalize()
        snn.snn_simulate(net.h, 50)   # kernel attributes are settled
        nets.append(net)
    a, b = nets
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        snn.snn_simulate(a.h, 50)
    with torch.cuda.stream(s):
        for _ in range(3):
            g.replay()
    for _ in range(3):
        snn.snn_simulate(b.h, 50)
    torch.cuda.synchronize()
    assert a.stats().t_now == b.stats().t_now == 200
    for x, y in zip((*a.read_state(), a.read_rb()), (*b.read_state(), b.read_rb())):
        assert np.array_equal(x, y)
    for net in nets:
        net.close()
