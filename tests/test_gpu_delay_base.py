"""Networks whose drawn delays start above the rule's lower end: window cells count
from the declared delay, the ring-buffer window from the drawn one.  The same
synapses given as an edge list (where both agree) give the same bits, static and
plastic, through the single calls and the cycle."""
import numpy as np
import pytest

from gpu_common import need_gpu, stream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("plastic", [0, 1], ids=["static", "plastic"])
@pytest.mark.parametrize("fmt", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("n,d_lo,d_hi,seed", [(24, 1, 31, 14), (40, 5, 30, 92), (9, 8, 28, 4)])
def test_declared_and_drawn_delays(n, d_lo, d_hi, seed, fmt, plastic):
    from paper_2109_12855_gb300 import snn
    n_i = n // 4
    rule = snn.conn_params(k_exc=1, k_inh=0, w_exc=900.0, w_inh=0.0, sd_exc=90.0,
                           d_lo=d_lo, d_hi=d_hi, seed=seed)

    def net_of(connect):
        p = snn.params(n_exc=n - n_i, n_inh=n_i, weight_format=fmt, seed=5,
                       nu_ext=40000.0, w_ext=60.0, n_slots=32)
        net = snn.Net(p, stream())
        if plastic:
            snn.snn_set_stdp(net.h, snn.stdp_params(lam=0.05, alpha=0.1, mu=0.4,
                                                    w_max=5000.0, w0=900.0))
        connect(net)
        net.finalize()
        return net

    with net_of(lambda x: x.connect_fixed_indegree(rule)) as a:
        rp, tg, dl, w = a.read_store()
        assert int(dl.min()) == d_lo + 3   # (what this is about: seeds picked so)
        D = a.stats().interval
        rows = np.repeat(np.arange(n), np.diff(rp.astype(np.int64)))
        with net_of(lambda x: x.connect_edges(rows, tg, dl, w.astype(np.float64))) as b:
            for net in (a, b):
                for _ in range(40):
                    snn.snn_update(net.h, snn.SNN_T_DEVICE, D)
                    snn.snn_deliver_pending(net.h)
                snn.snn_simulate(net.h, 405)
            sa, sb = a.stats(), b.stats()
            assert sa.error_flags == sb.error_flags == 0
            assert sa.spikes == sb.spikes > 0
            assert sa.events_delivered == sb.events_delivered > 0
            for x, y in zip((*a.read_state(), a.read_rb(), a.read_weights()),
                            (*b.read_state(), b.read_rb(), b.read_weights())):
                assert x.tobytes() == y.tobytes()
