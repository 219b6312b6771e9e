"""Bounds-checked build: the one-launch cycle and the vector additions of the
deliveries check what they read and add, too.  A store with corrupted records runs
through snn_simulate's cycle as through the single calls: the records are skipped,
SNN_ERRF_CHECK is raised, state and ring buffer agree bit for bit.

Runs only in a process that loaded the checked library (SNN_CHECKED=1, as
tests/test_gpu_checked_paths.py starts it)."""
import os

import numpy as np
import pytest

from gpu_common import need_gpu, stream

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(os.environ.get("SNN_CHECKED") != "1",
                                 reason="needs the bounds-checked library")]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    from paper_2109_12855_gb300 import snn
    assert snn.snn_checked()


@pytest.mark.parametrize("fmt,sd", [(0, 0.0), (0, 0.1), (1, 0.0), (1, 0.1), (1, 0.3)],
                         ids=["fp32-uniform", "fp32", "bf16-uniform", "bf16-integer",
                              "bf16-joined"])
def test_corrupt_records_in_the_cycle(fmt, sd):
    from paper_2109_12855_gb300 import snn
    n, steps = 3000, 205
    nets = []
    for _ in range(2):
        p = snn.params(n_exc=2400, n_inh=600, weight_format=fmt, seed=3,
                       nu_ext=27000.0)
        w = p.w_ext = snn.snn_psc_weight_for_psp(p, 0.1)
        net = snn.Net(p, stream())
        net.connect_fixed_indegree(snn.conn_params(
            k_exc=160, k_inh=40, w_exc=w, w_inh=-5 * w, sd_exc=sd * w,
            sd_inh=5 * sd * w, d_lo=10, d_hi=20, seed=41))
        net.finalize()
        rp = net.read_store()[0].astype(np.int64)
        for row in range(0, n, 10):      # one record of every tenth row
            at = int(rp[row] + (rp[row + 1] - rp[row]) // 2)
            if rp[row + 1] > rp[row]:
                snn.snn_debug_poke_record(net.h, at, (row // 10) % 2,
                                          n + 7 if (row // 10) % 2 == 0 else 27)
        nets.append(net)
    a, b = nets
    before = a.stats().kernel_launches
    snn.snn_simulate(a.h, steps)
    assert a.stats().kernel_launches - before == 1
    left = steps
    while left > 0:
        snn.snn_update(b.h, snn.SNN_T_DEVICE, min(10, left))
        snn.snn_deliver_pending(b.h)
        left -= 10
    sa, sb = a.stats(), b.stats()
    assert sa.error_flags == sb.error_flags == snn.SNN_ERRF_CHECK
    assert sa.spikes == sb.spikes > 1000
    for x, y in zip((*a.read_state(), a.read_rb()), (*b.read_state(), b.read_rb())):
        assert x.tobytes() == y.tobytes()
    for net in nets:
        net.close()


@pytest.mark.parametrize("n_sp", [40, 1500, 9000])
@pytest.mark.parametrize("fmt,sd", [(0, 0.0), (0, 0.1), (1, 0.0), (1, 0.1)],
                         ids=["fp32-uniform", "fp32", "bf16-uniform", "bf16-integer"])
def test_corrupt_records_in_lists(fmt, sd, n_sp):
    """Callers' lists of each length, with the records poked and with the same
    synapses left out of the network."""
    import workloads as W
    from paper_2109_12855_gb300 import snn
    n = 600
    src, tgt, d, _ = W.random_edges(n, 40000, 5, 9, seed=4)
    g = np.random.Generator(np.random.PCG64(1))
    w = g.normal(20.0, 1.0, len(src)) if sd else np.full(len(src), 20.0)
    s, t = W.random_spikes(n, n_sp, 0, 5, seed=n_sp)

    def net_of(keep):
        p = snn.params(n_exc=n, n_inh=0, weight_format=fmt)
        net = snn.Net(p, stream())
        net.connect_edges(src[keep], tgt[keep], d[keep], w[keep])
        net.finalize()
        return net

    with net_of(np.ones(len(src), bool)) as a:
        rp, tg, dl, ww = a.read_store()
        rows = np.repeat(np.arange(n), np.diff(rp.astype(np.int64)))
        bad = np.arange(17, len(rows), 61)
        for k, at in enumerate(bad):
            snn.snn_debug_poke_record(a.h, int(at), k % 2, 29 if k % 2 else n + 7)
        ok = np.ones(len(rows), bool)
        ok[bad] = False
        p = snn.params(n_exc=n, n_inh=0, weight_format=fmt)
        with snn.Net(p, stream()) as b:
            b.connect_edges(rows[ok].astype(np.uint32), tg[ok], dl[ok],
                            ww[ok].astype(np.float64))
            b.finalize()
            for net in (a, b):
                net.deliver(s, t.astype(np.int32))
            assert a.stats().error_flags == snn.SNN_ERRF_CHECK
            assert b.stats().error_flags == 0
            np.testing.assert_allclose(a.read_rb(), b.read_rb(), rtol=2e-6, atol=0)
