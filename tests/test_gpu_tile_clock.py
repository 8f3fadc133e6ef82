"""GPU: register tiles take the boundary data of the time one step per launch
takes them at, also where the clock has passed the whole numbers of FP32."""
import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run_from(clock, time_block, chunks):
    """A ramped plate from rest, its device clock (the one 64-bit word of the
    workspace that counts the steps) put to `clock` first."""
    import torch
    from paper_2208_04088_gb300 import _native as N
    wl = W.square_plate(48, 0)
    wl.bcs[1] = W.bc(W.TRACTION, (7e-4, 3e-4), W.RAMP, 3.0e7)
    s = N.Solver(N.desc_from_workload(wl, time_block=time_block))
    base = s.workspace.data_ptr() % 8
    words = s.workspace[(8 - base) % 8:]
    words = words[:words.numel() // 8 * 8].view(torch.int64)
    s.step(37)
    s.sync()
    at = words == 37
    s.step(5)
    s.sync()
    at &= words == 42
    assert int(at.sum()) == 1
    s.reset()
    words[at] = clock
    for c in chunks:
        s.step(c)
    s.sync()
    F = s.fields_host()
    assert int(words[at]) == clock + sum(chunks)
    s.close()
    return F


@pytest.mark.parametrize("clock", [0, 2 ** 24 - 6, 2 ** 24 + 2, 2 ** 24 + 3])
def test_ramp_beyond_exact_fp32_clock(clock):
    a = _run_from(clock, 1, [61])
    b = _run_from(clock, 0, [61])
    c = _run_from(clock, 0, [3, 8, 16, 34])
    assert np.abs(a["u"]).max() > 0
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k], b[k]), k
        assert np.array_equal(a[k], c[k]), k
