"""The two-step kernel's plan: which lattices it takes, as lbm_steps_per_pass says, and the
plans of several cells per warp and of one pass per launch, against the one-step kernels."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402


def passes(wl, **kw):
    lat = lbm.lattice_for(wl, **kw)
    try:
        lat.init_fields(*wl.initial_fields())
        before = lat.launch_count()
        lat.step(64)
        n = lat.launch_count() - before
        assert n == (2 if lat.steps_per_pass() == 2 else 64) or kw
        return lat.steps_per_pass()
    finally:
        lat.close()


def test_steps_per_pass():
    wl = W.random_case(400, 200, seed=1, bc=W.BC_FREESLIP, D=20, U=0.04)
    assert passes(wl) == 2
    assert passes(wl, bounce=lbm.LBM_BOUNCE_INTERPOLATED) == 2
    assert passes(wl, kernel=lbm.LBM_KERNEL_TMA) == 1
    assert passes(wl, kernel=lbm.LBM_KERNEL_TMA_WAVE) == 1
    assert passes(wl, ctas_per_sm=1) == 1
    for storage in (lbm.LBM_F16_OFS, lbm.LBM_BF16_SR, lbm.LBM_F64):
        assert passes(wl, storage=storage) == 1
    # a body over a third of the width: more force slots than the plan's region holds
    assert passes(W.random_case(800, 400, seed=1, bc=W.BC_FREESLIP, D=300, U=0.04)) == 1
    b = lbm.Batch([wl, wl])
    try:
        assert b.steps_per_pass() == 2
        b.set_kernel(lbm.LBM_KERNEL_TMA)
        assert b.steps_per_pass() == 1
    finally:
        b.close()


def compare(wl, steps):
    out = []
    for kernel in (lbm.LBM_KERNEL_DIRECT, lbm.LBM_KERNEL_AUTO):
        lat = lbm.lattice_for(wl, kernel=kernel)
        try:
            assert lat.steps_per_pass() == (2 if kernel == lbm.LBM_KERNEL_AUTO else 1)
            lat.init_fields(*wl.initial_fields())
            lat.step(steps)
            lat.sync()
            out.append((lat.get_populations(), lat.forces_raw()))
        finally:
            lat.close()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert np.array_equal(out[0][1], out[1][1])


# 1,301 and 2,001 windows for 2,432 warps: several bands per window, several cells per warp
@pytest.mark.parametrize("nx,ny", [(78_000, 48), (120_000, 31)])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_ZOUHE], ids=["periodic", "zouhe"])
def test_several_cells_per_warp(nx, ny, bc):
    compare(W.random_case(nx, ny, seed=3, bc=bc, D=8, U=0.04), 14)


def test_one_pass_per_launch():
    # just above 16M nodes: three passes, each a launch, so the buffers change on the host
    compare(W.random_case(4200, 4000, seed=2, bc=W.BC_FREESLIP, D=40, U=0.04), 7)
