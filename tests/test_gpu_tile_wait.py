"""GPU: waits inside the register tiles that run out are reported, never passed
over."""
import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

from helpers import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wl", [W.hole_plate(1024, 512, 64.0, 0),
                                W.edge_crack(600, 150, 0, lam_over_mu=0.8)],
                         ids=lambda w: f"{w.name}_{w.lam:.2g}")
@pytest.mark.parametrize("limit", [1, 300, 1000, 2000, 4000, 10 ** 5])
def test_short_wait_limit_times_out_or_changes_nothing(wl, limit):
    """A limit of about the time a copy takes or the block's warps wait for one
    another: a run either ends with the fields of one step per launch or reports
    LBM_ERR_TIMEOUT, and the handle then runs on after a reset."""
    from paper_2208_04088_gb300 import _native as N
    ref = run_gpu(wl, 43, time_block=1)
    s = N.Solver(N.desc_from_workload(wl))
    assert s.info()["time_block"] > 1
    N.lbm_set_wait_limit(s.h, limit)
    s.step(43)
    try:
        s.sync()
    except N.LbmError as e:
        assert e.status == N.LBM_ERR_TIMEOUT
        N.lbm_set_wait_limit(s.h, 10 ** 9)
        s.reset()
        s.step(43)
        s.sync()
    got = s.fields_host()
    s.close()
    for k in ("u", "v", "sigma"):
        assert np.array_equal(got[k], ref[k]), k
