"""Pooling, upsampling and their gradients, eight channels per access and one:
the same bits as the operation written out in torch, at sizes and strides that
take either kernel."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import nn  # noqa: E402


def image(N, H, W, C, stride, offset, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((N, H, W, stride), device="cuda", generator=g).bfloat16()[..., offset:offset + C]


def children(x):  # the four pixels of each 2 x 2 block, in the kernels' order
    x = x.float()
    return x[:, ::2, ::2], x[:, ::2, 1::2], x[:, 1::2, ::2], x[:, 1::2, 1::2]


# (small image H, W, C, channel stride, first channel): vectors; one vector per row;
# more than one block per row; a channel count, a stride and an offset that are not
# multiples of eight
SHAPES = [(2, 3, 5, 32, 96, 64), (1, 1, 1, 8, 8, 0), (1, 4, 67, 256, 384, 0), (2, 3, 5, 12, 24, 0), (1, 6, 10, 8, 12, 0),
          (1, 6, 10, 8, 24, 4)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_bits(shape):
    N, H, W, C, S, O = shape
    small, big = image(N, H, W, C, S, O, 1), image(N, 2 * H, 2 * W, C, S, O, 2)
    mask, old = image(N, 2 * H, 2 * W, C, S, O, 3), image(N, 2 * H, 2 * W, C, S, O, 4)
    a, b, c, d = children(big)

    y = image(N, 2 * H, 2 * W, C, S, O, 5)
    nn.upsample2(small, S, y, S, N, H, W, C)
    assert torch.equal(y, small.repeat_interleave(2, 1).repeat_interleave(2, 2))
    y = image(N, H, W, C, S, O, 5)
    nn.upsample2_bwd(big, S, y, S, N, H, W, C)
    assert torch.equal(y, (((a + b) + c) + d).bfloat16())
    y = image(N, H, W, C, S, O, 5)
    nn.avgpool2(big, S, y, S, N, 2 * H, 2 * W, C)
    assert torch.equal(y, (0.25 * (((a + b) + c) + d)).bfloat16())
    for acc in (False, True):
        for m in (None, mask):
            y = old.clone(memory_format=torch.preserve_format) if S == C else image(N, 2 * H, 2 * W, C, S, O, 4)
            nn.avgpool2_bwd(small, S, y, S, N, 2 * H, 2 * W, C, accumulate=acc, mask=m, ms=S if m is not None else 0)
            want = 0.25 * small.float().repeat_interleave(2, 1).repeat_interleave(2, 2)
            if m is not None:
                want = torch.where(m.float() > 0, want, torch.zeros_like(want))
            if acc:
                want = want + old.float()
            assert torch.equal(y, want.bfloat16()), (acc, m is not None)


@pytest.mark.parametrize("cout", [32, 96, 256])
def test_bias_gradient(cout):
    # P = 2 * 37 * 133 pixels: fewer and more than a block's lanes; the sum of P
    # floats in float: P * 2^-24 of the sum of magnitudes bounds any order
    N, H, W = 2, 37, 133
    x, gy = image(N, H, W, 32, 32, 0, 1), image(N, H, W, cout, cout + 8, 8, 2)
    gw, gb = torch.zeros((cout, 3, 3, 32), device="cuda"), torch.zeros(cout, device="cuda")
    nn.conv3x3_wgrad(x, 32, gy, cout + 8, gw, gb, N, H, W, 32, cout)
    g = gy.double().reshape(-1, cout)
    assert torch.all((gb.double() - g.sum(0)).abs() <= N * H * W * 2.0 ** -24 * g.abs().sum(0))
