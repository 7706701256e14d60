"""Batches with enough rows of 128 pixels per SM for the convolution's folded kernels, the
third CTA slot and the transposed stores (from 3 and 16 rows per SM on) against the same
images one at a time, which stay below: the products of an output are added in the same
order, so the results are equal bit for bit.  The rows per CTA do not divide the heights,
so runs cross images and bands of columns."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr()) if t is not None else None


def _rand(shape, seed, scale=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (scale * torch.randn(shape, generator=g, device="cuda")).bfloat16()


MANY = [(23, 107, 128), (12, 103, 256), (7, 128, 384)]   # 2461, 2472 and 2688 rows
SOME = [(5, 101, 128)]                                   # 505 rows


@pytest.mark.parametrize("dgrad", [0, 1])
@pytest.mark.parametrize("cout", [16, 32, 64, 128])
@pytest.mark.parametrize("cin", [16, 32, 64, 128])
@pytest.mark.parametrize("nb,h,w", MANY + SOME)
def test_batch_is_its_images(nb, h, w, cin, cout, dgrad):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    x = _rand((nb, h, w, cin), 1)
    x[nb // 2, h // 2, 5, 3] = float("inf")
    wt = _rand((9, cin, cout) if dgrad else (9, cout, cin), 2, 0.1)
    bias = None if dgrad else torch.linspace(-1, 1, cout, device="cuda")
    whole, parts = (torch.full((nb, h, w, cout), 7.0, dtype=torch.bfloat16, device="cuda")
                    for _ in range(2))
    assert L.lb_nn_conv3x3(_p(x), _p(wt), _p(bias), _p(whole), nb, h, w, cin, cout, 1 - dgrad,
                           dgrad, None) == 0
    for k in range(nb):
        assert L.lb_nn_conv3x3(_p(x[k]), _p(wt), _p(bias), _p(parts[k]), 1, h, w, cin, cout,
                               1 - dgrad, dgrad, None) == 0
    nan = torch.isnan(whole)
    assert torch.equal(nan, torch.isnan(parts)) and torch.equal(whole[~nan], parts[~nan])
    assert L.lb_nn_status() == abi.LB_OK
