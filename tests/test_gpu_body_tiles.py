"""Bodies that cross a row-tile boundary of some kernel shape but none of another: a
lattice is accepted wherever the body lies, and every kernel gives the same forces."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402


def run(wl, **kw):
    lat = lbm.lattice_for(wl, **kw)
    try:
        lat.init_fields(*wl.initial_fields())
        lat.step(3)
        lat.sync()
        return lat.get_populations(), lat.forces_raw()
    finally:
        lat.close()


# nodes per row tile: 256 (direct), 512, 640, 768, 832 and, in the 16-bit kernels,
# twice as many; each centre is a multiple of one of them
@pytest.mark.parametrize("xc", [512, 640, 768, 832, 1024, 1280])
@pytest.mark.parametrize("storage", [lbm.LBM_F32, lbm.LBM_F16_OFS], ids=["f32", "f16"])
def test_body_on_a_tile_boundary(xc, storage):
    wl = W.Workload(name="boundary", nx=1600, ny=60, D=20, xc=xc, yc=30, U=0.05, tau=0.6, perturb=0.05, seed=xc)
    ref = run(wl, storage=storage, kernel=lbm.LBM_KERNEL_DIRECT)
    runs = [dict(), dict(kernel=lbm.LBM_KERNEL_TMA), dict(kernel=lbm.LBM_KERNEL_TMA_BULK)]
    runs += [dict(kernel=lbm.LBM_KERNEL_TMA, shape=s) for s in [(16, 1, 4), (10, 2, 4), (12, 2, 4), (13, 2, 3)]]
    for kw in runs:
        got = run(wl, storage=storage, **kw)
        assert np.array_equal(got[0].view(np.uint8), ref[0].view(np.uint8)), kw
        assert np.array_equal(got[1], ref[1]), kw
