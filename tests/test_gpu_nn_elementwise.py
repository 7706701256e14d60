"""Pooling, upsampling, ReLU mask, add, residual loss and input expansion against
torch on the same BF16 values: channel counts with and without the 16-byte path,
buffers off the 16-byte grid, single rows and columns, odd widths.  Every result
is one rounding of an FP32 value formed in a stated order, so outputs are equal
bit for bit; the loss is an FP32 sum (1e-5)."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr())


def _bf(shape, seed, off=0):
    """BF16 values `off` elements past an allocation's start."""
    n = 1
    for v in shape:
        n *= v
    g = torch.Generator(device="cpu").manual_seed(seed)
    buf = torch.zeros(n + off, dtype=torch.bfloat16, device="cuda")
    t = buf[off:].view(shape)
    t.copy_(torch.randn(shape, generator=g))
    return t


SHAPES = [(1, 1, 1, 8), (2, 3, 5, 16), (1, 7, 33, 24), (3, 2, 4, 12), (1, 5, 6, 1), (1, 130, 3, 64)]


@pytest.mark.parametrize("off", [0, 1, 8])
@pytest.mark.parametrize("shape", SHAPES)
def test_pool_and_upsample(shape, off):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    nb, h, w, c = shape
    co, fi = _bf(shape, 1, off), _bf((nb, 2 * h, 2 * w, c), 2, off)
    f = fi.float()
    quads = ((f[:, 0::2, 0::2] + f[:, 0::2, 1::2]) + f[:, 1::2, 0::2]) + f[:, 1::2, 1::2]
    spread = lambda t: t.repeat_interleave(2, 1).repeat_interleave(2, 2)
    for call, size, src, want in (
            (L.lb_nn_pool2, (2 * h, 2 * w, c, 0), fi, (0.25 * quads).bfloat16()),
            (L.lb_nn_pool2, (2 * h, 2 * w, c, 1), co, spread((0.25 * co.float()).bfloat16())),
            (L.lb_nn_up2, (h, w, c, 0), co, spread(co)),
            (L.lb_nn_up2, (h, w, c, 1), fi, quads.bfloat16())):
        out = _bf(want.shape, 3, off)
        assert call(_p(src), _p(out), nb, *size, None) == 0
        assert torch.equal(out, want)


@pytest.mark.parametrize("n,off", [(8, 0), (4096, 0), (4096, 3), (4097, 0), (7, 0)])
def test_mask_and_add(n, off):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    a, b, out = _bf((n,), 1, off), _bf((n,), 2, off), _bf((n,), 3, off)
    b[::5] = 0.0
    assert L.lb_nn_relu_mask(_p(a), _p(b), _p(out), n, None) == 0
    assert torch.equal(out, torch.where(b > 0, a, torch.zeros_like(a)))
    assert L.lb_nn_add(_p(a), _p(b), _p(out), n, None) == 0
    assert torch.equal(out, (a.float() + b.float()).bfloat16())


@pytest.mark.parametrize("n,c,off", [(1, 16, 0), (300, 16, 0), (300, 16, 4), (257, 1, 0),
                                     (33, 24, 0), (40, 5, 0)])
def test_loss_and_expansion(n, c, off):
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    y, dy = _bf((n, c), 1), _bf((n, c), 2, off)
    g = torch.Generator(device="cpu").manual_seed(3)
    base, tgt = (torch.randn(n, generator=g).cuda() for _ in range(2))
    loss = torch.zeros(1, device="cuda")
    assert L.lb_nn_mse(_p(y), c, _p(tgt), _p(base), n, _p(loss), _p(dy), None) == 0
    d = base + y[:, 0].float() - tgt
    want = torch.zeros_like(dy)
    want[:, 0] = (2.0 * d / n).bfloat16()
    assert torch.equal(dy, want)
    ref = (d.double() ** 2).mean().item()
    assert abs(loss.item() / ref - 1.0) < 1e-5
    out = _bf((n, c), 5, off)
    assert L.lb_nn_expand(_p(base), _p(tgt), 0.3, _p(out), c, n, None) == 0
    want = torch.zeros_like(out)
    for k, v in enumerate((base, torch.full_like(base, 0.3), base - tgt)[:c]):
        want[:, k] = v.bfloat16()
    assert torch.equal(out, want)


@pytest.mark.parametrize("cin,cout,h", [(16, 16, 8), (16, 32, 64), (64, 128, 16)])
def test_bias_and_weight_sums_add_up(cin, cout, h):
    """The chunk sums of the weight gradient, reduced by eight warps: accumulated
    twice, dw doubles (FP32 sums of a few hundred chunks: 1e-5 of the largest)."""
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    x, dy = _bf((2, h, 128, cin), 1), _bf((2, h, 128, cout), 2)
    nbytes = L.lb_nn_wgrad_workspace(2, h, 128, cin, cout)
    ws = torch.empty(nbytes // 4, device="cuda")
    dw, db = torch.zeros((9, cout, cin), device="cuda"), torch.zeros(cout, device="cuda")
    for _ in range(2):
        assert L.lb_nn_conv3x3_wgrad(_p(x), _p(dy), _p(dw), _p(db), 2, h, 128, cin, cout, _p(ws),
                                     nbytes, None) == 0
    xd, yd = x.double(), dy.double()
    for tap in range(9):
        s = torch.roll(xd, (1 - tap // 3, 1 - tap % 3), (1, 2))
        ref = 2.0 * torch.einsum("bhwn,bhwc->nc", yd, s)
        assert (dw[tap].double() - ref).abs().max() < 1e-5 * ref.abs().max() * 10
    assert (db.double() - 2 * yd.sum((0, 1, 2))).abs().max() < 1e-5 * yd.abs().sum() / cout


@pytest.mark.parametrize("nb,h,w,c", [(1, 1, 1, 8), (2, 3, 5, 24), (1, 70, 9, 64), (3, 2, 40, 32)])
def test_chains_equal_the_single_calls(nb, h, w, c):
    """The chained passes against the calls that they replace, bit for bit."""
    from paper_2212_07848_gb300 import abi
    L = abi.load()
    small, big = (nb, h, w, c), (nb, 2 * h, 2 * w, c)
    sa, sb, fa, fb, act, facts = (_bf(s, i) for i, s in enumerate((small, small, big, big, small, big)))
    act[:, :, ::2] = 0.0
    new = lambda t: torch.full_like(t, 7.0)
    n, m = sa.numel(), fa.numel()
    # gradient of the upsampling, then the mask
    s, z, s2, z2 = (new(sa) for _ in range(4))
    assert L.lb_nn_up2(_p(fa), _p(s), nb, h, w, c, 1, None) == 0
    assert L.lb_nn_relu_mask(_p(s), _p(act), _p(z), n, None) == 0
    assert L.lb_nn_up2_relu_bwd(_p(fa), _p(act), _p(s2), _p(z2), nb, h, w, c, None) == 0
    assert torch.equal(s2, s) and torch.equal(z2, z)
    assert L.lb_nn_up2_relu_bwd(_p(fa), _p(act), None, _p(s2), nb, h, w, c, None) == 0
    assert torch.equal(s2, z)
    # gradient of the pooling, with and without a second branch, then the mask
    t, f, f2 = (new(fa) for _ in range(3))
    assert L.lb_nn_pool2(_p(sa), _p(t), nb, 2 * h, 2 * w, c, 1, None) == 0
    for add in (None, fb):
        if add is not None:
            assert L.lb_nn_add(_p(t), _p(add), _p(t), m, None) == 0
        assert L.lb_nn_relu_mask(_p(t), _p(facts), _p(f), m, None) == 0
        assert L.lb_nn_pool2_relu_bwd(_p(sa), None if add is None else _p(add), _p(facts), _p(f2),
                                      nb, 2 * h, 2 * w, c, None) == 0
        assert torch.equal(f2, f)
    # sum, then the upsampling
    assert L.lb_nn_add(_p(sa), _p(sb), _p(s), n, None) == 0
    assert L.lb_nn_up2(_p(s), _p(f), nb, h, w, c, 0, None) == 0
    assert L.lb_nn_add_up2(_p(sa), _p(sb), _p(s2), _p(f2), nb, h, w, c, None) == 0
    assert torch.equal(s2, s) and torch.equal(f2, f)
    # refused: channel counts and buffers off the 16-byte grid
    off = _bf(big, 9, 1)
    assert L.lb_nn_up2_relu_bwd(_p(fa), _p(act), None, _p(s2), nb, h, w, c - 4, None) != 0
    assert L.lb_nn_add_up2(_p(sa), _p(sb), None, _p(off), nb, h, w, c, None) != 0
