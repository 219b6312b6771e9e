"""An interval's own list through every way a tile adds up runs: counts of uniform
weights in halves of a word and, where an interval could bring a cell more than
65,535 events, in a word each or as integer weights; fixed point; and element by
element (counted cells, weights without exact sums).  Neurons without a
refractory period make the bound large on a small net: in-degree x steps of an
interval.

Tolerance: 1e-5 sum|w| per cell against Algorithm REF in 64 bits (the repository's
reading of relative error under E/I cancellation); the exact sums differ from it by
one rounding of a cell and one of the ring buffer."""
import numpy as np
import pytest

import oracle as O
from gpu_common import fixed_net, need_gpu

pytestmark = pytest.mark.gpu
S = 32


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


FORMS = [
    # fmt, spread, in-degree, counted
    pytest.param(0, 0.0, 4360, 0, id="fp32-counts-65400"),
    pytest.param(0, 0.0, 4370, 0, id="fp32-wide-65550"),
    pytest.param(1, 0.0, 4370, 0, id="bf16-uniform-65550"),
    pytest.param(1, 0.1, 4370, 0, id="bf16-spread"),
    pytest.param(0, 0.1, 300, 0, id="fp32-spread"),
    pytest.param(0, 0.0, 4370, 1, id="fp32-counted"),
    pytest.param(1, 0.1, 300, 1, id="bf16-spread-counted"),
]


@pytest.mark.parametrize("fmt,sd,k,counted", FORMS)
@pytest.mark.parametrize("words", [0, 2])
@pytest.mark.parametrize("firing", [1, 30, 65])
def test_own_list(fmt, sd, k, counted, words, firing):
    from paper_2109_12855_gb300 import snn
    n_e, n_i, k_e = 52, 13, k * 4 // 5
    w_e, w_i = 22.4058, -112.029
    net, cp = fixed_net(n_e, n_i, k_e, k - k_e, w_e, w_i, 15, 18, 9, fmt=fmt,
                        sd_e=sd * w_e, sd_i=-sd * w_i, acc_words=words,
                        count_events=counted, t_ref=0.0, v_reset=0.0)
    store = O.build_fixed_indegree(cp)
    n = n_e + n_i
    with net:
        # enough current for a spike in most steps, in the first `firing` neurons
        V = np.full(n, 30.0)
        V[np.random.Generator(np.random.PCG64(firing)).permutation(n)[firing:]] = 0.0
        J = np.where(V > 0, 4e6, 0.0)
        net.write_state(V, J, J, np.zeros(n, np.int32))
        snn.snn_update(net.h, snn.SNN_T_DEVICE, 15)
        src, t = np.zeros(n * 15, np.uint32), np.zeros(n * 15, np.int32)
        m = snn.snn_read_pending(net.h, src, t)
        src, t = src[:m], t[:m]
        assert m > 5 * firing        # (several spikes of a neuron in an interval)
        snn.snn_deliver_pending(net.h)
        rb_o, cnt_o, absw, ev_o = O.deliver_ref(store, S, src, t.astype(np.int64))
        st = net.stats()
        assert st.error_flags == 0 and st.events_delivered == ev_o
        err = np.abs(net.read_rb().astype(np.float64) - rb_o)
        assert np.all(err <= 1e-5 * absw + 1e-12), float(err.max())
        if counted:
            assert np.array_equal(net.read_counts().astype(np.int64),
                                  cnt_o.astype(np.int64))
