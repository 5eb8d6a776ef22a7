"""The start from device fields with infinite and NaN values: the formula's answer,
in which a zero component of c times an infinite velocity is NaN."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def central(f, axis):
    return 0.5 * (np.roll(f, -1, axis) - np.roll(f, 1, axis))


@pytest.mark.parametrize("noneq", [False, True], ids=["equilibrium", "with-noneq"])
@pytest.mark.parametrize("storage", [lbm.LBM_F32, lbm.LBM_F64], ids=["f32", "f64"])
def test_nonfinite_velocities(storage, noneq):
    nx, ny, U, tau = 64, 30, 0.05, 0.6
    r = np.ones((ny, nx), np.float32)
    u = np.full((ny, nx), U, np.float32)
    v = np.zeros((ny, nx), np.float32)
    u[8, 10], v[8, 20], u[8, 30], v[20, 40] = np.inf, -np.inf, np.nan, np.nan
    u[20, 10], v[20, 10] = np.inf, np.inf
    u[20, 20], r[20, 30], r[15, 50] = 3e38, np.inf, np.nan
    dev = [torch.from_numpy(t).cuda() for t in (r, u, v)]
    torch.cuda.synchronize()
    lat = lbm.Lattice(nx, ny, tau, U, mask=None, bc=W.BC_PERIODIC, D_ref=10.0, storage=storage)
    try:
        lbm.lbm_init_fields_device(lat.h, *(t.data_ptr() for t in dev), noneq)
        got = lat.get_populations()
    finally:
        lat.close()
    with np.errstate(all="ignore"):
        r, u, v = (t.astype(np.float64) for t in (r, u, v))
        ux, uy, vx, vy = central(u, 1), central(u, 0), central(v, 1), central(v, 0)
        want = np.empty((9, ny, nx))
        for k in range(9):
            cu = CX[k] * u + CY[k] * v
            f = WT[k] * r * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (u * u + v * v))
            if noneq:
                q = (CX[k] ** 2 - 1 / 3) * ux + (CY[k] ** 2 - 1 / 3) * vy + CX[k] * CY[k] * (uy + vx)
                f = f - 3.0 * (tau - 1.0) * WT[k] * r * q
            want[k] = f - WT[k] * (1 + 3 * CX[k] * U + 4.5 * CX[k] ** 2 * U * U - 1.5 * U * U)
        want = want.astype(got.dtype)
    inner = (slice(None), slice(2, -2), slice(2, -2))
    got, want = got[inner], want[inner]
    assert np.array_equal(np.isnan(got), np.isnan(want))
    for sign in (np.inf, -np.inf):
        assert np.array_equal(got == sign, want == sign)
