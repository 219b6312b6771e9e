"""The plastic rule's power of two (the PTX instruction ex2.approx.ftz.f32,
used where the result is a normal float) against exp2f and against 2^x in
64 bits, over the range that the rule's condition leaves it: exponents
mu log2(w) for weights above 1e-30 and mu up to 1 (from -100), trace decays
down to 2^-125, and both ends of the normal floats.

Tolerance: two units in the last place, the bound that the PTX ISA and the
CUDA C++ guide publish for the two, is a relative error of at most 2^-22."""
import numpy as np
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _ranges():
    g = np.random.Generator(np.random.PCG64(1))
    return {
        "decays": -g.uniform(0.0, 125.0, 1 << 20),
        "weights": np.log2(np.exp(g.uniform(np.log(1e-30), np.log(1e4), 1 << 20)))
        * g.uniform(0.0, 1.0, 1 << 20),
        "near zero": g.normal(0.0, 1e-3, 1 << 18),
        "whole": np.arange(-126.0, 128.0),
        "ends": np.concatenate([np.linspace(-126.0, -124.0, 4097),
                                np.linspace(126.0, 127.99, 4097),
                                [0.0, -0.0, 1e-38, -1e-38]]),
    }


@pytest.mark.parametrize("name", ["decays", "weights", "near zero", "whole", "ends"])
def test_power_of_two_is_as_near_as_exp2f(name):
    import torch
    from paper_2109_12855_gb300 import snn
    x = _ranges()[name].astype(np.float32)
    d = torch.from_numpy(x).cuda()
    a, b = torch.empty_like(d), torch.empty_like(d)
    snn.snn_probe_exp2(d, a, b)
    exact = np.exp2(x.astype(np.float64))
    ea = np.abs(a.cpu().numpy() / exact - 1.0)
    eb = np.abs(b.cpu().numpy() / exact - 1.0)
    assert ea.max() <= 2.0 ** -22
    assert eb.max() <= 2.0 ** -22
    assert ea.max() <= eb.max() and ea.mean() <= eb.mean()


def test_probe_rejects_bad_arguments():
    import torch
    from paper_2109_12855_gb300 import snn
    x = torch.zeros(8, device="cuda")
    with pytest.raises(ValueError):
        snn.snn_probe_exp2(x, x.clone(), torch.zeros(8))
    with pytest.raises(ValueError):
        snn.snn_probe_exp2(x, x.clone(), torch.zeros(4, device="cuda"))
    e = torch.zeros(0, device="cuda")
    with pytest.raises(snn.SnnError):
        snn.snn_probe_exp2(e, e, e)
