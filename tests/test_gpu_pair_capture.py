"""lbm_step under a caller's stream capture: a graph of an even number of steps can be
launched again and again, as it starts and ends in the same buffer."""
import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402

CASES = [W.random_case(181, 50, 1, W.BC_FREESLIP, D=10), W.random_case(400, 120, 3, W.BC_ZOUHE, D=20)]


def direct(wl, n):
    lat = lbm.lattice_for(wl, kernel=lbm.LBM_KERNEL_DIRECT)
    try:
        lat.init_fields(*wl.initial_fields())
        lat.step(n)
        lat.sync()
        return lat.get_populations(), lat.forces_raw()
    finally:
        lat.close()


def capture(stream, step, n):
    """Graph of step(n) on the stream (the library makes no other call there)."""
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        step(n)
    return g


@pytest.mark.parametrize("steps", [2, 4, 6, 34, 70])
def test_replays_of_a_lattice(steps):
    wl, replays = CASES[1], 3
    lat = lbm.lattice_for(wl)
    try:
        lat.init_fields(*wl.initial_fields())
        g = capture(lat.stream, lat.step, steps)
        with torch.cuda.stream(lat.stream):
            for _ in range(replays):
                g.replay()
        lat.sync()
        got = lat.get_populations(), lat.forces_raw()
    finally:
        lat.close()
    want = direct(wl, steps * replays)
    assert np.array_equal(got[0].view(np.uint32), want[0].view(np.uint32))
    assert np.array_equal(got[1], want[1])


def test_replays_of_a_batch():
    steps, replays = 6, 3
    b = lbm.Batch(CASES)
    try:
        b.init_all()
        g = capture(b.stream, b.step, steps)
        with torch.cuda.stream(b.stream):
            for _ in range(replays):
                g.replay()
        b.sync()
        for c, wl in enumerate(CASES):
            want = direct(wl, steps * replays)
            assert np.array_equal(b.get_populations(c).view(np.uint32), want[0].view(np.uint32))
            assert np.array_equal(b.forces_raw(c), want[1])
    finally:
        b.close()
