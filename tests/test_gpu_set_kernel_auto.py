"""lbm_set_kernel(AUTO) gives back what a new lattice has: the two-step kernel."""
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402


def launches(target, n):
    before = target.launch_count()
    target.step(n)
    target.sync()
    return target.launch_count() - before


def test_lattice_and_batch():
    wl = W.random_case(181, 50, 1, W.BC_FREESLIP, D=10)
    lat = lbm.lattice_for(wl)
    lat.init_fields(*wl.initial_fields())
    batch = lbm.Batch([wl, wl])
    batch.init_all()
    try:
        for target, set_kernel in ((lat, lbm.lbm_set_kernel), (batch, lbm.lbm_batch_set_kernel)):
            assert launches(target, 64) == 2
            set_kernel(target.h, lbm.LBM_KERNEL_TMA)
            assert launches(target, 64) == 64
            set_kernel(target.h, lbm.LBM_KERNEL_AUTO)
            assert launches(target, 64) == 2
        # one CTA per SM stays the default of an explicit kernel
        lbm.lbm_set_kernel(lat.h, lbm.LBM_KERNEL_TMA)
        assert lat.kernel_info()["ctas_per_sm"] == 1
    finally:
        lat.close()
        batch.close()
