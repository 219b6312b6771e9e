"""Kernels of one net that follow each other without the host waiting: the
update that comes directly after a one-launch cycle reads the state and the
spike statistics that the cycle left, whether it comes through snn_update or
through a snn_simulate of a single interval, captured or not."""
import numpy as np
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _net(stream, n, k, fmt, sd):
    from paper_2109_12855_gb300 import snn
    n_i, k_i = n // 5, k // 5
    p = snn.params(n_exc=n - n_i, n_inh=n_i, weight_format=fmt, seed=21,
                   nu_ext=27000.0)
    w = p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
    net = snn.Net(p, stream)
    net.connect_fixed_indegree(snn.conn_params(
        k_exc=k - k_i, k_inh=k_i, w_exc=w, w_inh=-5 * w, sd_exc=sd * w,
        sd_inh=5 * sd * w, d_lo=10, d_hi=20, seed=5))
    net.finalize()
    return net


def _single(net, steps, sync):
    from paper_2109_12855_gb300 import snn
    while steps > 0:
        snn.snn_update(net.h, snn.SNN_T_DEVICE, min(10, steps))
        if sync:
            snn.snn_sync(net.h)
        snn.snn_deliver_pending(net.h)
        if sync:
            snn.snn_sync(net.h)
        steps -= 10


def _result(net):
    from paper_2109_12855_gb300 import snn
    st = net.stats()
    return [*net.read_state(), net.read_rb(),
            *snn.snn_read_spike_stats(net.h, net.n),
            np.array([st.t_now, st.spikes, st.events_delivered, st.error_flags])]


def _equal(a, b):
    for x, y in zip(_result(a), _result(b)):
        assert x.tobytes() == y.tobytes()


@pytest.mark.parametrize("n,k,fmt,sd", [
    pytest.param(1250, 100, 0, 0.0, id="20-tiles"),
    pytest.param(20003, 400, 1, 0.1, id="every-sm"),
    pytest.param(110001, 200, 1, 0.0, id="one-wave-update"),
])
def test_update_after_cycle(n, k, fmt, sd):
    import torch
    from paper_2109_12855_gb300 import snn
    s = torch.cuda.Stream()
    with _net(s.cuda_stream, n, k, fmt, sd) as a, \
            _net(s.cuda_stream, n, k, fmt, sd) as b:
        for _ in range(12):
            snn.snn_simulate(a.h, 205)       # one launch, a short last interval
            _single(a, 10, False)            # an update right behind it
            snn.snn_simulate(a.h, 50)
            snn.snn_simulate(a.h, 5)         # fewer than two intervals: the
            snn.snn_simulate(a.h, 30)        # separate kernels, and a cycle again
        for _ in range(12):
            for steps in (205, 10, 50, 5, 30):
                _single(b, steps, True)
        _equal(a, b)


def test_update_after_cycle_in_a_captured_graph():
    import torch
    from paper_2109_12855_gb300 import snn
    s = torch.cuda.Stream()
    a, b = (_net(s.cuda_stream, 20003, 400, 1, 0.1) for _ in range(2))
    for net in (a, b):                       # kernel attributes are settled
        snn.snn_simulate(net.h, 50)
        snn.snn_simulate(net.h, 10)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        snn.snn_simulate(a.h, 50)
        snn.snn_simulate(a.h, 10)
    with torch.cuda.stream(s):
        for _ in range(10):
            g.replay()
    for _ in range(10):
        _single(b, 60, True)
    torch.cuda.synchronize()
    assert a.stats().t_now == b.stats().t_now
    for x, y in zip((*a.read_state(), a.read_rb()), (*b.read_state(), b.read_rb())):
        assert x.tobytes() == y.tobytes()
    for net in (a, b):
        net.close()
