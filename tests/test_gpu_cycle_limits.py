"""What snn_simulate's one-launch cycle does when something it counts on does
not hold (the conditions are made on the host, or by a wait with a short limit:
no launch faults or hangs)."""
import numpy as np
import pytest

from gpu_common import need_gpu, stream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _net(n=6001, k=300, fmt=1, sd=0.1):
    from paper_2109_12855_gb300 import snn
    n_i, k_i = n // 5, k // 5
    p = snn.params(n_exc=n - n_i, n_inh=n_i, weight_format=fmt, seed=8,
                   nu_ext=27000.0, spike_log_capacity=1 << 18)
    w = p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
    net = snn.Net(p, stream())
    net.connect_fixed_indegree(snn.conn_params(
        k_exc=k - k_i, k_inh=k_i, w_exc=w, w_inh=-5 * w, sd_exc=sd * w,
        sd_inh=5 * sd * w, d_lo=10, d_hi=20, seed=5))
    net.finalize()
    return net


def _state(net):
    return [*net.read_state(), net.read_rb()]


def test_wait_that_runs_out():
    """The call's launches end, the error is flagged, the clock is not moved,
    nothing runs on the broken state, and the net works again once its errors
    are cleared and a state is loaded."""
    from paper_2109_12855_gb300 import snn
    with _net() as a, _net() as b:
        for net in (a, b):
            snn.snn_simulate(net.h, 200)
        image = snn.snn_save_state(a.h)
        snn.snn_debug_cycle(a.h, snn.SNN_CYCLE_POLLS, 0)
        snn.snn_simulate(a.h, 10 * 600)          # three launches
        st = a.stats()
        assert st.error_flags == snn.SNN_ERRF_TIMEOUT
        assert st.t_now == 200
        # (reading the log empties it)
        assert len(a.read_spikes()[0]) == len(b.read_spikes()[0])
        broken = _state(a)
        snn.snn_debug_cycle(a.h, snn.SNN_CYCLE_POLLS, 1 << 24)
        snn.snn_simulate(a.h, 500)               # still flagged: does nothing
        assert a.stats().t_now == 200
        assert len(a.read_spikes()[0]) == 0
        for x, y in zip(broken, _state(a)):
            assert x.tobytes() == y.tobytes()
        snn.snn_clear_errors(a.h)
        snn.snn_load_state(a.h, image)
        for net in (a, b):
            snn.snn_simulate(net.h, 505)
        assert a.stats().error_flags == 0 and a.stats().t_now == b.stats().t_now == 705
        for x, y in zip(_state(a), _state(b)):
            assert x.tobytes() == y.tobytes()


@pytest.mark.parametrize("fmt,sd", [(0, 0.0), (0, 0.1), (1, 0.1)],
                         ids=["uniform", "fp32", "bf16"])
def test_missing_scales_are_flagged(fmt, sd):
    """The kernel finds no exact sums where the host had: the lists' events
    cannot be added up, and the net says so."""
    from paper_2109_12855_gb300 import snn
    with _net(2000, 200, fmt, sd) as net:
        snn.snn_simulate(net.h, 100)
        assert net.stats().error_flags == 0 and net.stats().spikes > 0
        snn.snn_debug_cycle(net.h, snn.SNN_CYCLE_UNSCALED, 1)
        snn.snn_simulate(net.h, 100)
        assert net.stats().error_flags == snn.SNN_ERRF_SCALES


@pytest.mark.parametrize("steps", [205, 35], ids=["graphs", "few-intervals"])
def test_refused_launch_runs_the_separate_kernels(steps):
    """A context with fewer SMs than the net has tiles refuses the cooperative
    launch: the call goes through the update and delivery kernels, to the same
    bits, and so does the next."""
    from paper_2109_12855_gb300 import snn
    with _net() as a, _net() as b:
        snn.snn_debug_cycle(a.h, snn.SNN_CYCLE_REFUSED, 1)
        for _ in range(2):
            before = a.stats().kernel_launches
            for net in (a, b):
                snn.snn_simulate(net.h, steps)
            assert a.stats().kernel_launches - before == 2 * -(-steps // 10)
        sa, sb = a.stats(), b.stats()
        assert sa.error_flags == sb.error_flags == 0
        assert (sa.t_now, sa.spikes, sa.events_delivered) == \
            (sb.t_now, sb.spikes, sb.events_delivered)
        for x, y in zip(_state(a), _state(b)):
            assert x.tobytes() == y.tobytes()


@pytest.mark.parametrize("most,launches", [(0, 2 * 41), (1, 41), (7, 6), (256, 1)])
def test_intervals_of_a_launch(most, launches):
    from paper_2109_12855_gb300 import snn
    with _net() as a, _net() as b:
        snn.snn_set_cycle(a.h, most)
        before = a.stats().kernel_launches
        for net in (a, b):
            snn.snn_simulate(net.h, 405)
        assert a.stats().kernel_launches - before == launches
        for x, y in zip(_state(a), _state(b)):
            assert x.tobytes() == y.tobytes()
        assert a.stats().t_now == b.stats().t_now == 405
        for bad in (-1, 257):
            with pytest.raises(snn.SnnError) as e:
                snn.snn_set_cycle(a.h, bad)
            assert e.value.code == snn.SNN_E_ARG


def test_options_are_checked():
    from paper_2109_12855_gb300 import snn
    with _net(500, 50) as net:
        for option, value in ((snn.SNN_CYCLE_POLLS, -1), (99, 0), (snn.SNN_CYCLE_REFUSED, 2),
                              (snn.SNN_CYCLE_POLLS, (1 << 24) + 1)):
            with pytest.raises(snn.SnnError) as e:
                snn.snn_debug_cycle(net.h, option, value)
            assert e.value.code == snn.SNN_E_ARG
