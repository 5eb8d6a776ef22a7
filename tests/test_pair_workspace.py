"""The two-step kernel's tables lie once in a batch, not in each of its cases (host only)."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def lbm():
    from paper_2605_02185_gb300 import _build, lbm
    _build.build()
    lbm.load_library()
    return lbm


def opts(lbm, **kw):
    o = lbm.lbm_opts_default()
    o.history_capacity = 1
    for k, v in kw.items():
        setattr(o, k, v)
    return o


def test_a_case_of_a_batch_costs_its_populations(lbm):
    case = dict(nx=64, ny=8, tau=0.6, U=0.05)
    o = opts(lbm)
    one, two = (lbm.lbm_batch_workspace_bytes([case] * n, [None] * n, o) for n in (1, 2))
    populations = 2 * 9 * 8 * 64 * 4
    assert two - one < populations + 64 * 1024
    # a single lattice may be given the two-step kernel later, so its workspace holds them
    single = opts(lbm, nx=64, ny=8, tau=0.6, U=0.05)
    assert lbm.lbm_workspace_bytes(single, None) - populations > 1 << 20
    assert two - 2 * populations > 1 << 20
