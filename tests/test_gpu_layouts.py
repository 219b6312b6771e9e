"""Split store layouts of the tiled delivery (uniform weights as counted
cells, integer, joined and FP32 weights): every layout delivers lists of every
form as Algorithm REF (the FP64 oracle) does, and reads back the store it was
built from.

Sizes sit at the edges of the 16-byte vectors a run is read in: runs of a few
synapses (several runs in one vector's span), of about one vector per lane,
and longer than the vectors loaded ahead; lists of one spike, of one batch of
run descriptors and of several, of more events a cell than 16-bit counts
hold, and spanning more steps than the window (global atomics).

Tolerance: 1e-5 sum|w| per cell (the repository's reading of relative error
under E/I cancellation), 1e-4 for the list whose cells take tens of thousands
of additions.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import fixed_net, need_gpu

pytestmark = pytest.mark.gpu
S = 32


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


FORMS = [
    # fmt, weight spread, d_lo, d_hi, acc_words
    pytest.param(0, 0.0, 15, 15, 0, id="fp32-uniform"),
    pytest.param(0, 0.1, 10, 20, 0, id="fp32-spread"),
    pytest.param(1, 0.0, 10, 20, 0, id="bf16-uniform"),
    pytest.param(1, 0.1, 10, 20, 0, id="bf16-integer"),
    pytest.param(1, 0.1, 1, 3, 2, id="bf16-two-word"),
    pytest.param(1, 0.3, 10, 12, 0, id="bf16-near-zero"),
]
# neurons, in-degree, tile width: runs of ~1, ~9 and ~300 synapses
SIZES = [(331, 20, 0), (601, 150, 37), (1203, 300, 1203)]


@pytest.mark.parametrize("fmt,sd,d_lo,d_hi,words", FORMS)
@pytest.mark.parametrize("n,k,tw", SIZES)
def test_lists_match_ref(fmt, sd, d_lo, d_hi, words, n, k, tw):
    from paper_2109_12855_gb300 import snn
    n_e = n * 4 // 5
    k_e = k * 4 // 5
    w_e, w_i = 22.4058, -112.029
    net, cp = fixed_net(n_e, n - n_e, k_e, k - k_e, w_e, w_i, d_lo, d_hi, 77,
                        fmt=fmt, sd_e=sd * w_e, sd_i=-sd * w_i, tile_width=tw,
                        acc_words=words, count_events=0)
    store = O.build_fixed_indegree(cp)
    span = min(d_lo, 15)
    lists = [(1, span, 1e-5), (57, span, 1e-5), (1100, span, 1e-5),
             (4500, span, 1e-5), (70000, span, 1e-4), (500, 45, 1e-5)]
    with net:
        for n_sp, steps, tol in lists:
            snn.snn_clear_rb(net.h)
            src, t = W.random_spikes(n, n_sp, 40, 40 + steps, seed=n_sp)
            ev = net.deliver(src, t.astype(np.int32))
            rb_o, _, absw, ev_o = O.deliver_ref(store, S, src, t)
            assert ev == ev_o
            err = np.abs(net.read_rb().astype(np.float64) - rb_o)
            assert np.all(err <= tol * absw + 1e-12), (n_sp, float(err.max()))


@pytest.mark.parametrize("fmt", [0, 1])
def test_uniform_edges_per_population(fmt):
    """An explicit edge list with one weight per population of sources is
    stored as counted cells; a single other weight anywhere is not lost."""
    from paper_2109_12855_gb300 import snn
    from gpu_common import stream
    n_e, n_i, m = 240, 60, 9001
    src, tgt, d, _ = W.random_edges(n_e + n_i, m, 2, 9, seed=5)
    for odd in (False, True):
        w = np.where(src < n_e, 3.5, -17.0)
        if odd:
            w[4321] = 2.25
        p = snn.params(n_exc=n_e, n_inh=n_i, weight_format=fmt)
        with snn.Net(p, stream()) as net:
            net.connect_edges(src, tgt, d, w)
            net.finalize()
            store = O.build_edges(n_e + n_i, src, tgt, d, w)
            s, t = W.random_spikes(n_e + n_i, 900, 0, 2, seed=6)
            net.deliver(s, t.astype(np.int32))
            rb_o, _, absw, _ = O.deliver_ref(store, S, s, t)
            assert np.all(np.abs(net.read_rb() - rb_o) <= 1e-5 * absw + 1e-12)
            assert sorted(net.read_store()[3].tolist()) == sorted(w.tolist())


@pytest.mark.parametrize("n_sp", [1, 1023, 1024, 2049, 4096, 4097])
@pytest.mark.parametrize("steps", [5, 40])
def test_lists_read_as_they_stand(n_sp, steps):
    """Device arrays around the longest list delivered without preparation:
    events counted, values as REF, a source outside the network skipped and
    flagged, steps far from the clock and spread past the window alike."""
    import torch
    from paper_2109_12855_gb300 import snn
    net, cp = fixed_net(400, 100, 40, 10, 20.0, -100.0, 10, 20, 7, fmt=0,
                        sd_e=2.0, sd_i=10.0, count_events=0)
    store = O.build_fixed_indegree(cp)
    src, t = W.random_spikes(500, n_sp, 1000, 1000 + steps, seed=n_sp)
    bad = np.concatenate([src, [500]]).astype(np.uint32)
    tb = np.concatenate([t, [1000]]).astype(np.int32)
    rb_o, _, absw, ev_o = O.deliver_ref(store, S, src, t)
    with net:
        for s, tt, flag in ((src, t, 0), (bad, tb, snn.SNN_ERRF_BAD_SOURCE)):
            snn.snn_clear_rb(net.h)
            ev = snn.snn_deliver(
                net.h, torch.from_numpy(s.view(np.int32).copy()).cuda(),
                torch.from_numpy(tt.astype(np.int32)).cuda())
            assert ev == ev_o
            assert np.all(np.abs(net.read_rb() - rb_o) <= 1e-5 * absw + 1e-12)
            assert net.stats().error_flags == flag


@pytest.mark.parametrize("n_sp,launches", [(4096, 1), (4097, 2)])
def test_launch_counts_around_the_longest_raw_list(n_sp, launches):
    """Both list entries count the kernels that they launch."""
    import torch
    from paper_2109_12855_gb300 import snn
    net, _ = fixed_net(400, 100, 40, 10, 20.0, -100.0, 15, 15, 7, fmt=0)
    src, t = W.random_spikes(500, n_sp, 1000, 1015, seed=n_sp)
    with net:
        s = torch.from_numpy(src.astype(np.int32)).cuda()
        tt = torch.from_numpy(t.astype(np.int32)).cuda()
        for deliver in (snn.snn_deliver, snn.snn_deliver_noalloc):
            before = net.stats().kernel_launches
            deliver(net.h, s, tt)
            assert net.stats().kernel_launches - before == launches
