"""Small lattices on streams of their own run at the same time: a launch of the two-step
kernel holds only the shared memory and registers of the warps it uses."""
import time

import numpy as np
import pytest

from paper_2605_02185_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2605_02185_gb300 import lbm  # noqa: E402


def seconds(lats, rounds=8, n=512):
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(rounds):
            for lat in lats:
                lat.step(n)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


# side by side: 1.3 times one lattice's time (four of 200 x 100) and 1.15 times (two of
# 400 x 200); one after another: 4 and 2 times
@pytest.mark.parametrize("size,count,limit", [((200, 100), 4, 2.5), ((400, 200), 2, 1.6)], ids=["200x100", "400x200"])
def test_lattices_overlap(size, count, limit):
    works = [W.random_case(*size, seed=k, bc=W.BC_FREESLIP, D=10, U=0.04) for k in range(count)]
    lats = [lbm.lattice_for(w) for w in works]
    try:
        for lat, w in zip(lats, works):
            lat.init_fields(*w.initial_fields())
        one = seconds(lats[:1])
        all_of_them = seconds(lats)
        for lat, w in zip(lats, works):  # and none disturbs another
            lat.init_fields(*w.initial_fields())
        for _ in range(3):
            for lat in lats:
                lat.step(70)
        for lat, w in zip(lats, works):
            lat.sync()
            ref = lbm.lattice_for(w, kernel=lbm.LBM_KERNEL_DIRECT)
            ref.init_fields(*w.initial_fields())
            ref.step(210)
            assert np.array_equal(lat.get_populations().view(np.uint32), ref.get_populations().view(np.uint32))
            ref.close()
        assert all_of_them < limit * one, (one, all_of_them)
    finally:
        for lat in lats:
            lat.close()
