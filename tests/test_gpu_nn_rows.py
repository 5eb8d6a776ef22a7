"""The row-marching convolution (8 to 96 channels) against the FP64 network
oracle on the same bfloat16 values (5e-3 of the output's scale: 2^-8 is the
bfloat16 step) and, on infinities, against the mma.sync kernels."""
import numpy as np
import pytest

from oracle import conv_oracle as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import nn  # noqa: E402

PAIRS = [(8, 32), (32, 8), (32, 32), (32, 64), (32, 96), (64, 32), (64, 64), (96, 32)]


@pytest.fixture(autouse=True)
def impl_reset():
    nn.status(reset=True)
    yield
    nn.set_conv_impl(nn.IMPL_AUTO)
    assert nn.status(reset=True) == 0  # no bounded wait gave up


def bf(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda().bfloat16()


def f64(t):
    return t.float().cpu().numpy().astype(np.float64)


# one pixel; one row, less than a tile; a tile, one pixel more and a ragged one;
# rows enough for every ring slot, several segments per CTA (many CTAs take one row
# of this many, and a long column is cut between CTAs)
@pytest.mark.parametrize("N,H,W", [(1, 1, 1), (2, 1, 20), (1, 9, 128), (2, 5, 129), (1, 3, 300), (1, 700, 260)])
@pytest.mark.parametrize("cin,cout", PAIRS)
def test_matches_oracle(cin, cout, N, H, W):
    rng = np.random.default_rng(cin + 3 * cout + W)
    xb = bf(rng.standard_normal((N, H, W, cin + 8)))  # channel slices of wider buffers
    x = xb[..., 8:]
    w = bf(rng.standard_normal((cout, 3, 3, cin)) / np.sqrt(9 * cin))
    b = torch.from_numpy(rng.standard_normal(cout).astype(np.float32)).cuda()
    m = bf(rng.standard_normal((N, H, W, cout)))
    ref = C.conv3x3(f64(x), f64(w), b.cpu().numpy())
    y = torch.full((N, H, W, cout + 16), 7.0, dtype=torch.bfloat16, device="cuda")
    nn.conv3x3_fwd(x, cin + 8, w, b, y[..., 8:], cout + 16, N, H, W, cin, cout, 1)
    assert torch.all(y[..., :8] == 7.0) and torch.all(y[..., 8 + cout:] == 7.0)
    got, want = f64(y[..., 8:8 + cout]), C.relu(ref)
    assert np.max(np.abs(got - want)) <= 5e-3 * max(np.max(np.abs(want)), 1e-30)
    nn.conv3x3_fwd(x, cin + 8, w, None, y[..., 8:], cout + 16, N, H, W, cin, cout, 0, mask=m, ms=cout)
    got, want = f64(y[..., 8:8 + cout]), C.relu_grad(f64(m), ref - b.cpu().numpy())
    assert np.max(np.abs(got - want)) <= 5e-3 * max(np.max(np.abs(want)), 1e-30)


@pytest.mark.parametrize("cin,cout", [(8, 32), (32, 8), (32, 32)])
def test_infinities_stay_where_they_reach(cin, cout):
    rng = np.random.default_rng(5)
    x = rng.standard_normal((1, 7, 140, cin))
    x[0, 3, 60, 2], x[0, 0, 0, 1], x[0, 6, 139, 0] = np.inf, -np.inf, np.nan
    x = bf(x)
    w = bf(rng.standard_normal((cout, 3, 3, cin)))
    out = []
    for impl in (nn.IMPL_AUTO, nn.IMPL_MMA_SYNC):
        nn.set_conv_impl(impl)
        y = torch.empty((1, 7, 140, cout), dtype=torch.bfloat16, device="cuda")
        nn.conv3x3_fwd(x, cin, w, None, y, cout, 1, 7, 140, cin, cout, 0)
        out.append(y.float())
    for test in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(test(out[0]), test(out[1]))


@pytest.mark.parametrize("cin,cout", [(8, 32), (32, 8)])
def test_eight_channels_are_refused_by_name(cin, cout):
    x = torch.zeros((1, 2, 16, cin), dtype=torch.bfloat16, device="cuda")
    w = torch.zeros((cout, 3, 3, cin), dtype=torch.bfloat16, device="cuda")
    y = torch.zeros((1, 2, 16, cout), dtype=torch.bfloat16, device="cuda")
    nn.set_conv_impl(nn.IMPL_TCGEN05)
    with pytest.raises(RuntimeError):
        nn.conv3x3_fwd(x, cin, w, None, y, cout, 1, 2, 16, cin, cout, 0)
