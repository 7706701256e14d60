"""The loss of a training iteration is the FP32 sum of one term per warp of 32 pixels.
With the same difference at every pixel all terms are equal, so the sum does not depend
on the order in which they arrive and has to be the sequential FP32 sum bit for bit
(another grouping of the pixels rounds to another value)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr()) if t is not None else None


@pytest.mark.parametrize("c,grad", [(16, True), (8, True), (16, False), (3, True), (3, False)])
@pytest.mark.parametrize("d", [0.3, 0.011, 0.0207])
def test_one_term_per_warp(d, c, grad):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    n = 1 << 18   # a pixel a thread
    f = np.float32
    term, expected = f(32) * (f(d) * f(d)) / f(n), f(0)
    for _ in range(n // 32):
        expected = f(expected + term)
    by_blocks = f(0)
    for _ in range(n // 256):
        by_blocks = f(by_blocks + f(8) * term)
    assert expected != by_blocks
    y = torch.zeros((n, c), dtype=torch.bfloat16, device="cuda")
    base = torch.full((n,), d, device="cuda")
    target, loss = torch.zeros(n, device="cuda"), torch.zeros(1, device="cuda")
    dy = torch.full_like(y, 7.0) if grad else None
    assert L.lb_nn_mse(_p(y), c, _p(target), _p(base), n, _p(loss), _p(dy), None) == 0
    assert loss.item() == float(expected)
    if grad:
        g = torch.zeros_like(y)
        g[:, 0] = float(f(2) * f(d) / f(n))
        assert torch.equal(dy, g)
