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


def _ordered(y, target, base, loss, grad=True):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    n, c = y.shape
    terms = torch.full((L.lb_nn_mse_terms(n) + 32,), 7.0, device="cuda")
    dy = torch.empty_like(y) if grad else None
    assert L.lb_nn_mse_ordered(_p(y), c, _p(target), _p(base), n, _p(loss), _p(terms), _p(dy),
                               None) == 0
    assert (terms[-32:] == 7.0).all()
    return terms[:-32].cpu().numpy(), dy


@pytest.mark.parametrize("n", [1, 33, 4096, 70001, 1 << 20, 8 * 512 * 512])
@pytest.mark.parametrize("kind", ["normal", "same", "powers", "sparse", "large", "nan"])
def test_terms_in_order(n, kind):
    """The loss is the sequential FP32 sum of the terms, also where chunks of them cannot be
    rounded ahead (a binade's end, halfway terms, infinities) and from a loss that is not 0."""
    g = torch.Generator(device="cuda").manual_seed(3)
    target, y = torch.zeros(n, device="cuda"), torch.zeros((n, 8), dtype=torch.bfloat16, device="cuda")
    base = 0.02 * torch.randn(n, generator=g, device="cuda")
    if kind == "same":
        base.fill_(0.0207)
    elif kind == "powers":     # terms on few bits: many halfway cases
        base = torch.exp2(torch.randint(-12, 4, (n,), generator=g, device="cuda").float())
    elif kind == "sparse":
        base *= (torch.rand(n, generator=g, device="cuda") < 1e-3)
    elif kind == "large":
        base = 1e18 * base
    elif kind == "nan":
        base[n // 2] = float("nan")
    for start in (0.0, 0.37, -0.01):
        loss = torch.full((1,), start, device="cuda")
        terms, dy = _ordered(y, target, base, loss)
        expected = np.cumsum(np.concatenate([[start], terms]).astype(np.float32), dtype=np.float32)[-1]
        got = np.float32(loss.item())
        assert got == expected or (np.isnan(got) and np.isnan(expected)), start
    from paper_2212_07848_gb300 import abi
    plain = torch.empty_like(dy)     # the gradient is lb_nn_mse's
    assert abi.load().lb_nn_mse(_p(y), 8, _p(target), _p(base), n, _p(loss), _p(plain), None) == 0
    assert torch.equal(dy.view(torch.int16), plain.view(torch.int16))


def test_training_loss_repeats():
    from paper_2212_07848_gb300 import surrogate as S
    net = S.SurrogateNet(128, 2)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((2, 128, 128, 16), generator=g, device="cuda").bfloat16()
    base = torch.randn((2, 128, 128), generator=g, device="cuda")
    net.forward(x)
    got = [net.loss_and_grad(x, base + 0.1 * torch.roll(base, 1, 2), base).item() for _ in range(20)]
    assert len(set(got)) == 1
