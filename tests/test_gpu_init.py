"""The start from device fields, f_eq (+ f_neq), against the formula in double.

About thirty double operations on terms of magnitude <= 1 (2^-48 of them in all),
then one rounding to the storage type (relative 2^-24 for float; 2^-23 allows for a
tie the operations' order turns)."""
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


def feq(rho, u, v):
    out = np.empty((9,) + np.shape(rho))
    for k in range(9):
        cu = CX[k] * u + CY[k] * v
        out[k] = WT[k] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u + v * v))
    return out


def gradient(f, fluid, axis):
    ok = np.pad(fluid, 1)
    p = np.pad(f, 1)
    s = np.roll
    lo, hi = (s(a, 1, axis)[1:-1, 1:-1] for a in (ok, p)), (s(a, -1, axis)[1:-1, 1:-1] for a in (ok, p))
    (okl, fl), (okh, fh) = lo, hi
    return np.where(okl & okh, 0.5 * (fh - fl), np.where(okh, fh - f, np.where(okl, f - fl, 0.0)))


@pytest.mark.parametrize("noneq", [False, True])
@pytest.mark.parametrize("storage", [lbm.LBM_F32, lbm.LBM_F64, lbm.LBM_BF16_OFS], ids=["f32", "f64", "bf16"])
@pytest.mark.parametrize("size", [(37, 23), (256, 61)], ids=["37x23", "256x61"])
def test_start_matches_formula(size, storage, noneq):
    nx, ny = size
    wl = W.random_case(nx, ny, seed=4, bc=W.BC_FREESLIP, D=8, U=0.05, tau=0.56)
    rng = np.random.default_rng(1)
    r = (1 + 0.02 * rng.standard_normal((ny, nx))).astype(np.float32)
    u = (0.05 + 0.02 * rng.standard_normal((ny, nx))).astype(np.float32)
    v = (0.02 * rng.standard_normal((ny, nx))).astype(np.float32)
    dev = [torch.from_numpy(t).cuda() for t in (r, u, v)]
    torch.cuda.synchronize()
    lat = lbm.lattice_for(wl, storage=storage)
    try:
        lbm.lbm_init_fields_device(lat.h, *(t.data_ptr() for t in dev), noneq)
        got = lat.get_populations()
    finally:
        lat.close()
    if storage == lbm.LBM_BF16_OFS:
        got = (got.astype(np.uint32) << 16).view(np.float32)
    fluid = wl.mask() == 0
    r, u, v = (t.astype(np.float64) for t in (r, u, v))
    f = feq(r, u, v)
    if noneq:
        ux, uy, vx, vy = (gradient(t, fluid, a) for t in (u, v) for a in (1, 0))
        for k in range(9):
            Q = (CX[k] ** 2 - 1 / 3) * ux + (CY[k] ** 2 - 1 / 3) * vy + CX[k] * CY[k] * (uy + vx)
            f[k] -= 3 * (wl.tau - 1) * WT[k] * r * Q
    want = f - feq(1.0, 0.05, 0.0)[:, None, None]
    err = np.abs(got.astype(np.float64) - want)[:, fluid]
    eps = {lbm.LBM_F32: 2.0 ** -23, lbm.LBM_F64: 2.0 ** -50, lbm.LBM_BF16_OFS: 2.0 ** -8}[storage]
    assert np.all(err <= eps * np.abs(want)[:, fluid] + 2.0 ** -47), err.max()
    assert np.all(got[:, ~fluid] == 0)
