"""Uniform weights that a float (or bfloat16) holds only as infinity, as not a
number, or near its largest value, where no exact sums exist: a cell gets what
its own events add up to, and cells without an event of such a weight keep
finite values, in a caller's list of either form and in the net's own lists.

The other population's weight is -1, whose sums are whole numbers below 2^24:
the comparison is exact."""
import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu, stream

pytestmark = pytest.mark.gpu
S = 32


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _expected(net, src, t, w_e, n_e):
    """Ring buffer from the store's own rows: counts per cell and population."""
    rp, tg, dl, _ = net.read_store()
    rp = rp.astype(np.int64)
    n = net.n
    cnt = np.zeros((2, S, n))
    for s, tt in zip(src.astype(np.int64), t.astype(np.int64)):
        a, b = rp[s], rp[s + 1]
        np.add.at(cnt[int(s >= n_e)], ((tt + dl[a:b]) % S, tg[a:b]), 1.0)
    with np.errstate(invalid="ignore", over="ignore"):
        e = np.where(cnt[0] > 0, (cnt[0] * w_e).astype(np.float32), 0.0)
        return (e - cnt[1]).astype(np.float32)


@pytest.mark.parametrize("fmt", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("w_e", [np.inf, 1e39, np.nan, 3.2e38])
def test_uniform_weights_beyond_the_scales(fmt, w_e):
    from paper_2109_12855_gb300 import snn
    n_e, n_i = 400, 100
    p = snn.params(n_exc=n_e, n_inh=n_i, weight_format=fmt)
    with snn.Net(p, stream()) as net:
        # (not a number: alone, so that no other weight gives the sums a scale)
        net.connect_fixed_indegree(snn.conn_params(
            k_exc=8, k_inh=0 if np.isnan(w_e) else 4, w_exc=w_e, w_inh=-1.0,
            d_lo=10, d_hi=20, seed=3))
        net.finalize()
        stored = net.read_store()[3]
        w = float(stored[np.argmax(~(stored < 0))])
        g = np.random.Generator(np.random.PCG64(2))
        for n_sp, lo in ((40, n_e), (1, 0), (60, 0), (5000, n_e)):
            src = g.integers(lo, n_e + n_i, n_sp).astype(np.uint32)
            if n_sp == 60:
                src = np.arange(n_e + n_i - 60, n_e + n_i, dtype=np.uint32)
                src[::9] = 3 * np.arange(7)      # a few excitatory ones
            t = g.integers(0, 10, n_sp).astype(np.int32)
            snn.snn_clear_rb(net.h)
            net.deliver(src, t)
            np.testing.assert_array_equal(net.read_rb(), _expected(net, src, t, w, n_e))


@pytest.mark.parametrize("fmt", [0, 1], ids=["fp32", "bf16"])
def test_own_spikes_with_infinite_weights(fmt):
    """Neurons pushed over the threshold: their interval's list goes the same
    way; only inhibitory ones fire, so every cell stays finite."""
    from paper_2109_12855_gb300 import snn
    n_e, n_i = 400, 100
    p = snn.params(n_exc=n_e, n_inh=n_i, weight_format=fmt, init_v_random=0)
    with snn.Net(p, stream()) as net:
        net.connect_fixed_indegree(snn.conn_params(
            k_exc=8, k_inh=4, w_exc=1e39, w_inh=-1.0, d_lo=10, d_hi=20, seed=3))
        net.finalize()
        V = np.zeros(n_e + n_i, np.float32)
        V[n_e:n_e + 30] = 25.0
        net.write_state(V, 0 * V, 0 * V, np.zeros(n_e + n_i, np.int32))
        snn.snn_update(net.h, snn.SNN_T_DEVICE, 10)
        snn.snn_deliver_pending(net.h)
        src = np.arange(n_e, n_e + 30)
        np.testing.assert_array_equal(
            net.read_rb(), _expected(net, src, 0 * src, np.inf, n_e))
