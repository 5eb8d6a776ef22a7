"""The row-marching convolution adds in the order of the kernels it stands in for: the
same bits as conv_tc_kernel, which takes smaller images of the same content, and, for 8
channels, as the mma.sync kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import nn  # noqa: E402


@pytest.fixture(autouse=True)
def impl_reset():
    nn.status(reset=True)
    yield
    nn.set_conv_impl(nn.IMPL_AUTO)
    assert nn.status(reset=True) == 0


def conv(x, w, mask=None):
    N, H, Wd, cin = x.shape
    cout = w.shape[0]
    y = torch.empty((N, H, Wd, cout), dtype=torch.bfloat16, device="cuda")
    nn.conv3x3_fwd(x, cin, w, None, y, cout, N, H, Wd, cin, cout, 0, mask=mask, ms=cout if mask is not None else 0)
    return y.view(torch.int16)


def inputs(N, H, Wd, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    x = torch.randn((N, H, Wd, cin), device="cuda", generator=g).bfloat16()
    w = torch.randn((cout, 3, 3, cin), device="cuda", generator=g).bfloat16()
    m = torch.randn((N, H, Wd, cout), device="cuda", generator=g).bfloat16()
    return x, w, m


@pytest.mark.parametrize("cin,cout", [(32, 32), (32, 64), (32, 96), (64, 32), (64, 64), (96, 32)])
def test_same_bits_as_the_tile_kernel(cin, cout):
    # 1,000 rows of two tiles: above every line of the rule; 100 of them: below
    x, w, m = inputs(1, 1000, 200, cin, cout)
    for mask in (None, m):
        big = conv(x, w, mask)
        for h in (0, 450, 900):
            part = slice(h, h + 100)
            small = conv(x[:, part].contiguous(), w, None if mask is None else mask[:, part].contiguous())
            # the cut's first and last rows see zeros in place of their neighbours
            lo, hi = (0 if h == 0 else 1), (100 if h == 900 else 99)
            assert torch.equal(small[:, lo:hi], big[:, h + lo:h + hi])


@pytest.mark.parametrize("N,H,Wd", [(1, 9, 128), (2, 31, 129), (1, 700, 260)])
@pytest.mark.parametrize("cin,cout", [(8, 32), (32, 8)])
def test_same_bits_as_mma_sync(cin, cout, N, H, Wd):
    x, w, m = inputs(N, H, Wd, cin, cout)
    for mask in (None, m):
        got = conv(x, w, mask)
        nn.set_conv_impl(nn.IMPL_MMA_SYNC)
        want = conv(x, w, mask)
        nn.set_conv_impl(nn.IMPL_AUTO)
        assert torch.equal(got, want)
