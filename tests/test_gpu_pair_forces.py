"""Forces of the two-step kernel: a row's links are summed to no fewer bits than a
double holds, also past the float range, so that the history equals the one-step
kernels' wherever a double sum is exact."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

TAU = 1e30  # a relaxation rate that leaves every population as it is: steps only move them


def run(nx, ny, mask, pops, steps, **kw):
    lat = lbm.Lattice(nx, ny, TAU, 0.0, mask=mask, bc=W.BC_PERIODIC, D_ref=10.0, **kw)
    try:
        lat.set_populations(pops, 1)
        lat.step(steps)
        return lat.get_populations(), lat.forces_raw(1, steps), lat.launch_count()
    finally:
        lat.close()


@pytest.mark.parametrize("bounce", [lbm.LBM_BOUNCE_HALFWAY, lbm.LBM_BOUNCE_INTERPOLATED], ids=["half", "interp"])
@pytest.mark.parametrize("seed", range(4))
def test_sums_a_double_holds_exactly(seed, bounce):
    # a 3 x 3 body, links' populations multiples of 2^-55 below 2^-8: any sum of its 36
    # links is exact in double, and needs more than the 48 bits of two floats.  The body's
    # circle lies so that every interpolated link's fraction is one half (q = 1/2 returns
    # the population itself).
    nx, ny = 96, 40
    rng = np.random.default_rng(seed)
    m = rng.integers(2 ** 23, 2 ** 24, (9, ny, nx)).astype(np.float64) * rng.choice([-1.0, 1.0], (9, ny, nx))
    pops = (m * np.where(rng.random((9, ny, nx)) < 0.5, 2.0 ** -32, 2.0 ** -55)).astype(np.float32)
    mask = np.zeros((ny, nx), np.uint8)
    x0 = 30 + seed
    mask[18:21, x0:x0 + 3] = 1
    pops[:, mask == 1] = 0
    kw = dict(bounce=bounce)
    if bounce == lbm.LBM_BOUNCE_INTERPOLATED:
        kw["body"] = (x0 + 1.0, 19.0, 1e-3)  # no link meets so small a circle: fractions of one half
    ref = run(nx, ny, mask, pops, 2, kernel=lbm.LBM_KERNEL_DIRECT, **kw)
    got = run(nx, ny, mask, pops, 2, **kw)
    assert got[2] == 2  # one pass and its sums
    assert np.array_equal(ref[0].view(np.uint32), got[0].view(np.uint32))
    assert np.array_equal(ref[1], got[1])


def test_sums_past_the_float_range():
    # opposite populations are equal, so the state at rest stays as it is; a lane's two
    # nodes over the body's top hold six links of 8e37
    nx, ny = 96, 40
    mask = np.zeros((ny, nx), np.uint8)
    mask[15:20, 30:37] = 1
    pops = np.zeros((9, ny, nx), np.float32)
    pops[[2, 4, 5, 6, 7, 8]] = 8e37
    pops[0] = -3.2e38
    pops[:, mask == 1] = 0
    ref = run(nx, ny, mask, pops, 2, kernel=lbm.LBM_KERNEL_DIRECT)
    got = run(nx, ny, mask, pops, 2)
    assert np.all(np.isfinite(ref[1]))
    assert np.array_equal(ref[1], got[1])


def test_infinite_links():
    nx, ny = 96, 40
    mask = np.zeros((ny, nx), np.uint8)
    mask[15:20, 30:37] = 1
    pops = np.zeros((9, ny, nx), np.float32)
    pops[4, 21, 33] = np.inf
    ref = run(nx, ny, mask, pops, 2, kernel=lbm.LBM_KERNEL_DIRECT)
    got = run(nx, ny, mask, pops, 2)
    assert not np.all(np.isfinite(ref[1]))
    assert np.array_equal(ref[1], got[1], equal_nan=True)


@pytest.mark.parametrize("bounce", [lbm.LBM_BOUNCE_HALFWAY, lbm.LBM_BOUNCE_INTERPOLATED], ids=["half", "interp"])
def test_wide_body(bounce):
    # about a thousand links below 0.1: a double sum in another order differs by less than
    # 1000 x 2^-53 of the sum of magnitudes, 2 x 1000 x 0.1
    wl = W.random_case(1601, 300, seed=7, bc=W.BC_FREESLIP, D=140, U=0.04)
    out = []
    for kernel in (lbm.LBM_KERNEL_DIRECT, lbm.LBM_KERNEL_AUTO):
        lat = lbm.lattice_for(wl, kernel=kernel, bounce=bounce)
        try:
            lat.init_fields(*wl.initial_fields())
            lat.step(70)
            lat.sync()
            out.append((lat.get_populations(), lat.forces_raw()))
        finally:
            lat.close()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert np.abs(out[0][1] - out[1][1]).max() <= 1000 * 2.0 ** -53 * 200


def test_batch_sums_past_the_float_range():
    wl = W.Workload(name="rest", nx=96, ny=40, D=8, xc=33, yc=18, U=0.0, tau=TAU, bc=W.BC_PERIODIC)
    mask = wl.mask()
    pops = np.zeros((9, 40, 96), np.float32)
    pops[[2, 4, 5, 6, 7, 8]] = 8e37
    pops[0] = -3.2e38
    pops[:, mask == 1] = 0
    ref = run(96, 40, mask, pops, 2, kernel=lbm.LBM_KERNEL_DIRECT)
    b = lbm.Batch([wl])
    try:
        lbm.lbm_set_populations(b.case(0), pops, 1)
        b.step(2)
        got = b.forces_raw(0, 1, 2)
    finally:
        b.close()
    assert np.all(np.isfinite(ref[1]))
    assert np.array_equal(ref[1], got)
