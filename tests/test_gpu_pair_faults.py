"""The two-step kernel's bounded waits.  A row of its cells that does not report its
passes (and a short wait limit) makes the neighbours' waits run out: the launch returns,
lbm_sync reports LBM_ERR_TIMEOUT, and a new state gives the one-step kernels' bits
again.  Nothing faults: the waits end by themselves."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

WAIT = 0.05


def direct(wl, n, **kw):
    lat = lbm.lattice_for(wl, kernel=lbm.LBM_KERNEL_DIRECT, **kw)
    try:
        lat.init_fields(*wl.initial_fields())
        lat.step(n)
        lat.sync()
        return lat.get_populations(), lat.forces_raw()
    finally:
        lat.close()


def times_out(target):
    with pytest.raises(lbm.LBMError) as e:
        target.sync()
    return e.value.code == lbm.LBM_ERR_TIMEOUT


def same(got, want):
    assert np.array_equal(got[0].view(np.uint32), want[0].view(np.uint32))
    assert np.array_equal(got[1], want[1])


# 2 steps: one pass, which waits for nothing, so the one-step kernel takes them
@pytest.mark.parametrize("steps", [2, 4, 64, 70])
@pytest.mark.parametrize("bounce", [lbm.LBM_BOUNCE_HALFWAY, lbm.LBM_BOUNCE_INTERPOLATED], ids=["half", "interp"])
@pytest.mark.parametrize("size,bc", [((301, 57), W.BC_FREESLIP), ((61, 30), W.BC_PERIODIC), ((800, 400), W.BC_ZOUHE)],
                         ids=["301x57", "61x30", "800x400"])
def test_lattice_times_out_and_recovers(size, bc, bounce, steps):
    wl = W.random_case(*size, seed=5, bc=bc, D=8)
    lat = lbm.lattice_for(wl, bounce=bounce)
    try:
        lat.init_fields(*wl.initial_fields())
        lbm.lbm_set_fault_injection(lat.h, 7, WAIT)
        lat.step(steps)
        assert times_out(lat)
        lbm.lbm_set_fault_injection(lat.h, -1, 0.0)
        lat.init_fields(*wl.initial_fields())
        lat.step(70)
        lat.sync()
        same((lat.get_populations(), lat.forces_raw()), direct(wl, 70, bounce=bounce))
    finally:
        lat.close()


def test_wait_limit_alone_keeps_the_kernel():
    wl = W.random_case(301, 57, seed=5, bc=W.BC_FREESLIP, D=8)
    lat = lbm.lattice_for(wl)
    try:
        lat.init_fields(*wl.initial_fields())
        lbm.lbm_set_fault_injection(lat.h, -1, 0.5)
        before = lat.launch_count()
        lat.step(64)
        lat.sync()
        assert lat.launch_count() - before == 2
        same((lat.get_populations(), lat.forces_raw()), direct(wl, 64))
    finally:
        lat.close()


def test_choosing_the_kernel_again_keeps_the_fault():
    wl = W.random_case(301, 57, seed=5, bc=W.BC_FREESLIP, D=8)
    lat = lbm.lattice_for(wl)
    try:
        lat.init_fields(*wl.initial_fields())
        lbm.lbm_set_fault_injection(lat.h, 7, WAIT)
        lat.set_kernel(lbm.LBM_KERNEL_AUTO)
        lat.step(64)
        assert times_out(lat)
    finally:
        lat.close()


@pytest.mark.parametrize("steps", [2, 64, 70])
def test_batch_times_out_and_recovers(steps):
    cases = [W.random_case(97, 33, 1, W.BC_FREESLIP, D=8), W.random_case(241, 59, 4, W.BC_MOVINGWALL, D=10),
             W.random_case(400, 120, 3, W.BC_ZOUHE, D=20)]
    b = lbm.Batch(cases)
    try:
        b.init_all()
        lbm.lbm_batch_set_fault_injection(b.h, 1, 11, WAIT)
        b.step(steps)
        assert times_out(b)
        lbm.lbm_batch_set_fault_injection(b.h, 1, -1, 0.0)
        b.init_all()
        b.step(70)
        b.sync()
        for c, wl in enumerate(cases):
            same((b.get_populations(c), b.forces_raw(c)), direct(wl, 70))
    finally:
        b.close()


def test_recovery_past_other_kernels():
    # timed out, then a new state while the library's choice does not run, and back
    wl = W.random_case(301, 57, seed=5, bc=W.BC_FREESLIP, D=8)
    lat = lbm.lattice_for(wl)
    try:
        lat.init_fields(*wl.initial_fields())
        start = lat.get_populations()
        lbm.lbm_set_fault_injection(lat.h, 7, WAIT)
        lat.step(70)
        assert times_out(lat)
        lbm.lbm_set_fault_injection(lat.h, -1, WAIT)
        lat.set_populations(start, 1)
        lat.step(1)
        lbm.lbm_set_fault_injection(lat.h, -1, 0.0)
        lat.step(69)
        lat.sync()
        want = direct(wl, 70)
        same((lat.get_populations(), lat.forces_raw(1)), (want[0], want[1][1:]))
    finally:
        lat.close()


def test_batch_recovery_through_its_cases():
    cases = [W.random_case(97, 33, 1, W.BC_FREESLIP, D=8), W.random_case(241, 59, 4, W.BC_MOVINGWALL, D=10)]
    b = lbm.Batch(cases)
    try:
        b.init_all()
        starts = [b.get_populations(c) for c in range(2)]
        lbm.lbm_batch_set_fault_injection(b.h, 0, 5, WAIT)
        b.step(64)  # 32 passes: the batch stays on the buffer it began in
        assert times_out(b)
        lbm.lbm_batch_set_fault_injection(b.h, 0, -1, 0.0)
        for c in range(2):
            lbm.lbm_set_populations(b.case(c), starts[c], 1)
        b.step(70)
        b.sync()
        for c, wl in enumerate(cases):
            want = direct(wl, 70)
            same((b.get_populations(c), b.forces_raw(c, 1)), (want[0], want[1][1:]))
    finally:
        b.close()


def test_batch_arguments():
    wl = W.random_case(97, 33, 1, W.BC_FREESLIP, D=8)
    b = lbm.Batch([wl])
    try:
        for c, tile, wait in ((1, 0, WAIT), (-1, 0, WAIT), (0, 10 ** 6, WAIT), (0, 0, 61.0)):
            with pytest.raises(lbm.LBMError) as e:
                lbm.lbm_batch_set_fault_injection(b.h, c, tile, wait)
            assert e.value.code == lbm.LBM_ERR_ARG
        b.set_kernel(lbm.LBM_KERNEL_DIRECT)
        with pytest.raises(lbm.LBMError):
            lbm.lbm_batch_set_fault_injection(b.h, 0, 0, WAIT)
    finally:
        b.close()
