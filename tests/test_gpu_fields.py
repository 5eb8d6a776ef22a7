"""Read-back of rho, u, v in float against the library's double moments of the
same stored populations.

The float kernel works in float pairs: a sum of at most ten terms of magnitude
<= 1 carries an error below 2^-44, the quotient's remainder is formed exactly, and
the result is rounded to float once (relative 2^-24, and 2^-23 allows for the tie
that the pair error may turn)."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

STORAGES = [lbm.LBM_F32, lbm.LBM_F16_OFS, lbm.LBM_BF16_OFS, lbm.LBM_F16_SR, lbm.LBM_BF16_SR, lbm.LBM_F64]


@pytest.mark.parametrize("storage", STORAGES, ids=["f32", "f16", "bf16", "f16sr", "bf16sr", "f64"])
# rows of 4-node groups, a remainder (one node per thread), one group per row, and an
# output that is not 16-byte aligned
@pytest.mark.parametrize("size,shift", [((256, 61), 0), ((257, 61), 0), ((40, 33), 0), ((128, 40), 1)],
                         ids=["256x61", "257x61", "40x33", "128x40-unaligned"])
def test_float_fields_match_double_moments(size, shift, storage):
    nx, ny = size
    wl = W.random_case(nx, ny, seed=9, bc=W.BC_FREESLIP, D=10, U=0.05)
    lat = lbm.lattice_for(wl, storage=storage)
    try:
        lat.init_fields(*wl.initial_fields())
        lat.step(20)
        want = lat.fields(np.float64)
        got = [torch.full((ny * nx + 2,), -7.0, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        lbm.lbm_fields_device(lat.h, *(t.data_ptr() + 4 * shift for t in got))
        torch.cuda.synchronize()
    finally:
        lat.close()
    for g, w in zip(got, want):
        g = g.cpu().numpy()
        assert np.all(g[:shift] == -7.0) and np.all(g[shift + nx * ny:] == -7.0)
        err = np.abs(g[shift:shift + nx * ny].reshape(ny, nx).astype(np.float64) - w)
        assert np.all(err <= 2.0 ** -23 * np.abs(w) + 2.0 ** -43), err.max()
