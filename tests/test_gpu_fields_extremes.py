"""Float read-back of populations with infinities, NaN and sums that leave the float
range: the same answer as the library's double moments rounded to float."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

INF, NAN, BIG, DEN = np.inf, np.nan, 3e38, 1e-40
# nine populations of one node each
NODES = [
    [INF, 0, 0, 0, 0, 0, 0, 0, 0], [0, INF, 0, 0, 0, 0, 0, 0, 0], [0, 0, -INF, 0, 0, 0, 0, 0, 0],
    [INF, -INF, 0, 0, 0, 0, 0, 0, 0], [0, 0, 0, 0, 0, NAN, 0, 0, 0],
    [BIG, BIG, 0, 0, 0, 0, 0, 0, 0], [0, BIG, BIG, -BIG, 0, -BIG, 0, 0, 0], [-BIG, 0, BIG, 0, BIG, 0, 0, 0, 0],
    [1e20, 1e19, 0, 0, 0, 0, 0, 0, 3e18], [2e37, -1e30, 4e30, 0, 0, 0, 0, 0, 0],
    [-1, 0, 0, 0, 0, 0, 0, 0, 0], [-1, DEN, 0, 0, 0, 0, 0, 0, 0], [-1, 0, 3e-39, 0, 0, 0, 0, 0, DEN],
    [-1, 1e-36, -1e-38, 0, 0, 0, 0, 0, 0], [0, 0, DEN, 0, 0, 0, 0, 0, 0], [0, 0, 2e-38, 0, -1e-38, 0, 0, 0, 0],
    [-2, 0, 0, 0, 0, 0, 0, 0, 0], [1e-3, 0, 1e-3, 0, -1e-3, 1e-12, 0, 0, 1e-17],
]


@pytest.mark.parametrize("nx", [256, 257], ids=["four-nodes-a-thread", "one-node"])
@pytest.mark.parametrize("U", [0.05, 0.0], ids=["moving", "rest"])
def test_extreme_populations(nx, U):
    ny = 20
    lat = lbm.Lattice(nx, ny, 0.6, U, mask=None, bc=W.BC_PERIODIC, D_ref=10.0)
    try:
        pops = np.zeros((9, ny, nx), np.float32)
        for i, node in enumerate(NODES):
            pops[:, 5 + i % 7, 7 + 11 * i] = node
        lat.set_populations(pops, 1)
        with np.errstate(over="ignore"):
            want = [w.astype(np.float32) for w in lat.fields(np.float64)]
        got = lat.fields(np.float32)
    finally:
        lat.close()
    for g, w in zip(got, want):
        odd = ~np.isfinite(w)
        assert np.array_equal(g[odd], w[odd], equal_nan=True), (g[odd], w[odd])
        ulp = np.spacing(np.abs(w[~odd])).astype(np.float64)
        assert np.all(np.abs(g[~odd].astype(np.float64) - w[~odd]) <= ulp)


def test_small_velocities_keep_their_digits():
    """A transverse velocity far below its terms: nine terms of 2^-9 down to 2^-56 whose
    sum a double holds exactly, so the float result is the double one (one ulp for the
    order of the two roundings)."""
    ny, nx = 24, 512
    rng = np.random.default_rng(7)
    big = rng.integers(2 ** 23, 2 ** 24, (4, ny, nx)) * 2.0 ** -32
    small = rng.integers(2 ** 23, 2 ** 24, (9, ny, nx)) * 2.0 ** -56
    pops = small.copy()
    # what cancels: 2 and 4 (up and down), 5 and 8, 6 and 7
    pops[2] = pops[4] = big[0]
    pops[5], pops[8] = big[1], big[1]
    pops[6] = small[6]
    pops[7] = small[7]
    lat = lbm.Lattice(nx, ny, 0.6, 0.0, mask=None, bc=W.BC_PERIODIC, D_ref=10.0)
    try:
        lat.set_populations(pops.astype(np.float32), 1)
        want = [w.astype(np.float32) for w in lat.fields(np.float64)]
        got = lat.fields(np.float32)
    finally:
        lat.close()
    assert np.abs(want[2]).max() < 1e-9
    for g, w in zip(got, want):
        assert np.all(np.abs(g.astype(np.float64) - w) <= np.spacing(np.abs(w)))
