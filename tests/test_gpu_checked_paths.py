"""The bounds-checked build over the paths that the production build takes: the
one-launch cycle, every layout and way of adding up runs, updates behind a cycle
(a child process loads libsnn_check.so); no net of the clean cases may have raised
SNN_ERRF_CHECK, and corrupted stores are caught."""
import pytest

from gpu_common import need_gpu
from test_gpu_checked import _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def test_clean_cycles_and_layouts_raise_no_check():
    rc, out = _run(["tests/test_gpu_cycle.py", "tests/test_gpu_cycle_order.py",
                    "tests/test_gpu_layouts.py", "tests/test_gpu_add_modes.py",
                    "tests/test_gpu_serve.py"])
    assert rc == 0, out
    assert "nets flagged by the bounds checks: 0" in out


def test_corrupt_stores_are_caught_in_cycles_and_vectors():
    rc, out = _run(["tests/test_gpu_checked_cycle.py"])
    assert rc == 3, out
    assert "17 passed" in out, out
