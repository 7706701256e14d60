"""A line of the autotuner's cache is taken by ensembles whose steps run the kernel that it
was measured for, and by no others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LN2 = float(np.log(2.0))


def _tuned(tau, cache, kernel=None):
    from paper_2212_07848_gb300 import abi
    from paper_2212_07848_gb300.ensemble import Ensemble
    e = Ensemble([(256, 256, -3.6, tau, 1e-6, LN2)] * 3, seed=3)
    if kernel is not None:
        e.set_kernel(getattr(abi, kernel))
    e.init(0.0)
    got = e.autotune(3, cache)
    e.close()
    return got


def test_one_line_for_each_kernel(tmp_path):
    cache = str(tmp_path / "tune.txt")
    lines = lambda: open(cache).read().splitlines()
    first = _tuned(1.0, cache)
    _tuned(0.8, cache)                          # the general path
    _tuned(1.0, cache, "LB_KERNEL_OVERLAP")     # the wide strips
    assert len({ln.split()[0] for ln in lines()}) == 3
    assert _tuned(1.0, cache) == first and len(lines()) == 3


def test_lines_of_removed_kernels_are_not_taken(tmp_path):
    """A key that names only the layouts of earlier kernels."""
    cache = str(tmp_path / "tune.txt")
    _tuned(1.0, cache)
    key = open(cache).read().split()[0]
    old = key.replace("|pair64|unit", "|hw")
    assert old != key
    with open(cache, "w") as f:
        f.write(f"{old} 47\n")
    assert _tuned(1.0, cache) != 47
