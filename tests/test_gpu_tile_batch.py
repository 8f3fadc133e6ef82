"""GPU: instances of a batch stepped in register tiles keep their own results
whatever else the batch holds."""
import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _desc(wl, **kw):
    """With a body force, so that every material node moves from the first step."""
    from paper_2208_04088_gb300 import _native as N
    if wl is None:  # a lattice without material
        d = N.Desc(np.zeros((200, 256), np.uint8), np.zeros(0, N.LINK_DTYPE),
                   [W.bc(W.DIRICHLET, (0.0, 0.0))], W.MU, W.MU, **kw)
    else:
        d = N.desc_from_workload(wl, **kw)
    d.c.force[0], d.c.force[1] = 3e-6, -2e-6
    return d


def _alone(wl, steps):
    from paper_2208_04088_gb300 import _native as N
    s = N.Solver(_desc(wl, time_block=1))
    s.step(steps)
    s.sync()
    F = s.fields_host()
    s.close()
    return F


def _same(a, b):
    return all(np.array_equal(a[k], b[k]) for k in ("u", "v", "sigma"))


@pytest.mark.parametrize("at", [0, 1, 2, None], ids=["first", "second", "last", "three"])
@pytest.mark.parametrize("side", [640, 1100], ids=["one_kernel", "two_kernels"])
def test_instance_without_material(side, at):
    """The one tile of a lattice without material has nothing to step; the block
    that takes it takes another tile behind it, of another instance (the batch
    has more tiles than the device has SMs), whose displacements must be its
    own.  48 steps replay whole launches of eight, 13 end in one of five."""
    from paper_2208_04088_gb300 import _native as N
    wls = [W.hole_plate(side, side, 40.5, 0), W.hole_plate(260, 250, 20.3, 0)]
    if at is None:
        wls = [None, wls[0], None, wls[1], None]
    else:
        wls.insert(at, None)
    b = N.Batch([_desc(w) for w in wls])
    assert b.info()["blocked_instances"] == len(wls)
    ref = {id(w): {n: _alone(w, n) for n in (48, 61)} for w in wls if w}
    t = 0
    for n in (48, 13):
        b.step(n)
        b.sync()
        t += n
        for k, w in enumerate(wls):
            got = b.fields_host(k)
            if w is None:
                assert not any(got[q].any() for q in ("u", "v", "sigma"))
            else:
                assert _same(got, ref[id(w)][t]), (k, t)
    b.close()


@pytest.mark.parametrize("lam", [1.0, 0.8], ids=["poisson", "nonpoisson"])
def test_launches_of_two_kernels_on_two_streams(lam):
    """Two handles whose launches are two kernels each, the second released by
    the blocks of the first, stepped beside one another: every launch has its own
    count of released blocks, back at zero when it ends."""
    import torch
    from paper_2208_04088_gb300 import _native as N
    wls = [W.edge_crack(1300, 300, 0, lam_over_mu=lam, ny=1260),
           W.hole_plate(1250, 1340, 130.5, 0, lam_over_mu=lam)]
    ref = []
    for w in wls:
        s = N.Solver(_desc(w, time_block=1))
        s.step(120)
        s.sync()
        ref.append(s.fields_host())
        s.close()
    ss = [N.Solver(_desc(w), stream=torch.cuda.Stream()) for w in wls]
    before = [s.info()["kernel_launches"] for s in ss]
    for n in (8, 5, 40, 64, 3):
        for s in ss:
            s.step(n)
    for s, b in zip(ss, before):
        s.sync()
        # 120 steps: as many launches as chunks of them need, two kernels in each
        assert s.info()["kernel_launches"] - b > 2 * (120 // s.info()["time_block"])
        assert s.info()["time_block"] > 1
    for s, r in zip(ss, ref):
        assert _same(s.fields_host(), r)
        s.close()
