"""The persistent convolution's folded form (an input row to its three output rows in
one MMA) against the per-tile kernel, and its input gradient against its forward on
mirrored weights: the products of an output are summed in the same order, so the
results are equal bit for bit.  Images of 2 and 3 rows, one to three rows a CTA, runs
that wrap the ring of accumulators and cross bands and images, values at infinity."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr())


def _rand(shape, seed, scale=1.0):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return (scale * torch.randn(shape, generator=g)).bfloat16().cuda()


SIZES = [(1, 2, 128), (2, 3, 256), (1, 97, 384), (3, 160, 256), (2, 768, 128)]


def _same(a, b):
    nan = torch.isnan(a)
    return torch.equal(nan, torch.isnan(b)) and torch.equal(a[~nan], b[~nan])


@pytest.mark.parametrize("cin,cout", [(32, 16), (32, 32), (32, 64), (64, 16), (64, 32), (64, 64)])
@pytest.mark.parametrize("nb,h,w", SIZES)
def test_forward(nb, h, w, cin, cout):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    x, wt = _rand((nb, h, w, cin), 1), _rand((9, cout, cin), 2, 0.1)
    x[0, h // 2, 5, 3] = float("inf")
    bias = torch.randn(cout, generator=torch.Generator().manual_seed(3)).cuda()
    ys = []
    for path in (2, 3):
        assert L.lb_nn_set_conv_path(path) == 0
        y = torch.full((nb, h, w, cout), 7.0, dtype=torch.bfloat16, device="cuda")
        rc = L.lb_nn_conv3x3(_p(x), _p(wt), _p(bias), _p(y), nb, h, w, cin, cout, 1, 0, None)
        assert L.lb_nn_set_conv_path(0) == 0
        assert rc == 0
        ys.append(y)
    assert _same(*ys)
    assert L.lb_nn_status() == abi.LB_OK


@pytest.mark.parametrize("cout", [16, 32, 64, 128])
@pytest.mark.parametrize("cin", [16, 32, 64, 128])
@pytest.mark.parametrize("nb,h,w", SIZES)
def test_input_gradient(nb, h, w, cin, cout):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    dy, wt = _rand((nb, h, w, cin), 4), _rand((9, cin, cout), 5, 0.1)
    mirrored = wt.flip(0).transpose(1, 2).contiguous()
    out = torch.full((2, nb, h, w, cout), 7.0, dtype=torch.bfloat16, device="cuda")
    assert L.lb_nn_conv3x3(_p(dy), _p(wt), None, _p(out[0]), nb, h, w, cin, cout, 0, 1, None) == 0
    assert L.lb_nn_conv3x3(_p(dy), _p(mirrored), None, _p(out[1]), nb, h, w, cin, cout, 0, 0,
                           None) == 0
    assert torch.equal(out[0], out[1])
    assert L.lb_nn_status() == abi.LB_OK


@pytest.mark.parametrize("cout", [16, 32, 64, 128])
@pytest.mark.parametrize("cin", [16, 32, 64, 128])
@pytest.mark.parametrize("nb,h,w", SIZES)
def test_weight_gradient(nb, h, w, cin, cout):
    """Whole numbers below 2^24 in every sum: equal to the FP64 sums."""
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    g = torch.Generator(device="cpu").manual_seed(6)
    x, dy = (torch.randint(-3, 4, (nb, h, w, c), generator=g).bfloat16().cuda() for c in (cin, cout))
    dw = torch.zeros((9, cout, cin), device="cuda")
    size = L.lb_nn_wgrad_workspace(nb, h, w, cin, cout)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    assert L.lb_nn_conv3x3_wgrad(_p(x), _p(dy), _p(dw), None, nb, h, w, cin, cout, _p(ws), size,
                                 None) == 0
    d = dy.double().reshape(-1, cout)
    for tap in range(9):
        s = torch.roll(x, (1 - tap // 3, 1 - tap % 3), (1, 2)).double().reshape(-1, cin)
        assert torch.equal(dw[tap].double(), d.t() @ s), tap
    assert L.lb_nn_status() == abi.LB_OK
