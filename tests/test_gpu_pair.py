"""The two-step kernel (two steps per pass, many passes per launch) against the
one-step kernels: identical bits in every population and force, at the edges of
its 60-column windows and of its cells, whatever the split into calls."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

BCS = [W.BC_FREESLIP, W.BC_PERIODIC, W.BC_ZOUHE, W.BC_MOVINGWALL]


def run(wl, chunks, **kw):
    lat = lbm.lattice_for(wl, **kw)
    try:
        lat.init_fields(*wl.initial_fields())
        for n in chunks:
            lat.step(n)
        lat.sync()
        return lat.get_populations(), lat.forces_raw(), lat.launch_count()
    finally:
        lat.close()


def same(a, b):
    assert np.array_equal(a[0].view(np.uint32), b[0].view(np.uint32)), "populations differ"
    assert np.array_equal(a[1], b[1]), "force histories differ"


@pytest.mark.parametrize("bounce", [lbm.LBM_BOUNCE_HALFWAY, lbm.LBM_BOUNCE_INTERPOLATED], ids=["half", "interp"])
@pytest.mark.parametrize("mrt", [0, 1], ids=["bgk", "mrt"])
@pytest.mark.parametrize("bc", BCS, ids=[W.BC_NAMES[b] for b in BCS])
# 58 .. 61 columns: the outlet as the last column of a window, just past it, and
# in the next window; 1601 x 300: cells of several rows
@pytest.mark.parametrize("size", [(58, 21), (59, 24), (60, 22), (61, 30), (120, 40), (1601, 300)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
def test_matches_one_step_kernel(size, bc, mrt, bounce):
    wl = W.random_case(*size, seed=size[0] + bc, bc=bc, D=min(30, size[1] // 3), U=0.04)
    kw = dict(collision=mrt, bounce=bounce)
    ref = run(wl, [74], kernel=lbm.LBM_KERNEL_DIRECT, **kw)
    got = run(wl, [1, 2, 5, 66], **kw)  # 66 = 32 passes and one more
    assert got[2] < ref[2] // 2  # the two-step kernel ran
    same(ref, got)


def test_more_cells_than_warps():
    # 2,500 windows of 60 columns on at most 152 x 16 = 2,432 warps
    wl = W.random_case(150_000, 24, seed=3, bc=W.BC_PERIODIC, D=8)
    same(run(wl, [9], kernel=lbm.LBM_KERNEL_DIRECT), run(wl, [9]))


def test_no_body_appends_zero_forces():
    lat = lbm.Lattice(130, 40, 0.7, 0.08, mask=None, bc=W.BC_PERIODIC, D_ref=10.0)
    lat.init_fields(np.ones((40, 130)), np.full((40, 130), 0.08), np.zeros((40, 130)))
    lat.step(70)
    lat.sync()
    F = lat.forces_raw()
    lat.close()
    assert F.shape == (71, 2) and np.all(F == 0.0)


def test_unstable_flow_is_reported():
    wl = W.random_case(157, 43, seed=4, bc=W.BC_FREESLIP, D=8)
    lat = lbm.lattice_for(wl)
    lat.init_fields(*wl.initial_fields())
    lat.step(4)
    pops, n = lat.get_populations(), lat.force_count()
    pops[5, 20, 30] = np.nan
    lat.set_populations(pops, n)
    lat.step(2)
    with pytest.raises(lbm.LBMError) as e:
        lat.sync()
    assert e.value.code == lbm.LBM_ERR_UNSTABLE
    lat.close()


@pytest.mark.parametrize("mrt", [0, 1], ids=["bgk", "mrt"])
def test_batch_matches_one_step_kernel(mrt):
    cases = [W.random_case(97, 33, 1, W.BC_FREESLIP, D=8), W.random_case(61, 45, 2, W.BC_PERIODIC, D=8),
             W.random_case(400, 120, 3, W.BC_ZOUHE, D=20), W.random_case(241, 59, 4, W.BC_MOVINGWALL, D=10)]
    b = lbm.Batch(cases, collision=mrt)
    try:
        b.init_all()
        for n in (3, 37, 70):
            b.step(n)
        b.sync()
        for c, wl in enumerate(cases):
            ref = run(wl, [110], kernel=lbm.LBM_KERNEL_DIRECT, collision=mrt)
            same(ref, (b.get_populations(c), b.forces_raw(c)))
    finally:
        b.close()
