"""GPU: register-tile stepping, the default of most lattices (several steps per
launch, lbm_tile.cu).  Per node it performs the one-step arithmetic, so its
fields must be bit-identical to time_block = 1 for every tile shape, at the
edges of tiles and lattices, and for any split of a run into calls (a launch
carries any number of steps up to LBM_TIME_BLOCK)."""
import dataclasses

import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

from helpers import run_gpu, run_gpu_tables

pytestmark = pytest.mark.gpu


def _with(wl, **kw):
    return dataclasses.replace(wl, **kw)


def _rules(nx, ny, lam=1.0):
    """Every kind of boundary condition, corner links of every pairing, ramps."""
    wl = W.hole_plate(nx, ny, 0.2 * min(nx, ny) + 0.3, 0, lam_over_mu=lam)
    wl.bcs = [W.bc(W.DIRICHLET, (2e-4, -1e-4)), W.bc(W.DIRICHLET, (0.0, 0.0)),
              W.bc(W.STRESS, (1e-3, -5e-4, 3e-4)), W.bc(W.PRESSURE, (-4e-4,), W.RAMP, 20.0),
              W.bc(W.TRACTION, (2e-4, 6e-4), W.RAMP, 11.0)]
    wl.edge_bc = (0, 2, 3, 4)
    wl.hole = (*wl.hole[:3], 1)
    return _with(wl, name=f"rules_{nx}x{ny}_lam{lam:.2g}")


# one ring exactly, one node more, odd sizes, a single column of rings, lattices
# whose plan takes each of the larger tiles
SIZES = [(2, 3), (32, 32), (33, 31), (49, 65), (64, 17), (5, 200), (131, 90), (333, 217)]


@pytest.mark.parametrize("lam", [1.0, W.CRACK_PAPER_LAM_OVER_MU], ids=["poisson", "nonpoisson"])
@pytest.mark.parametrize("wall_node", [False, True], ids=["extrapolate", "node"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_default_bit_identical_to_one_step(nx, ny, wall_node, lam):
    wl = _with(_rules(nx, ny, lam), wall_node=wall_node)
    a = run_gpu(wl, 45, time_block=1)
    for chunks in (None, [1, 2, 3, 5, 7, 6, 21]):
        b = run_gpu(wl, 45, chunks=chunks)
        assert b["info"]["time_block"] == (8 if lam == 1.0 else 4)
        for k in ("u", "v", "sigma"):
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("wl", [W.hole_plate(1030, 517, 61.3, 0),
                                _with(W.centre_crack(100, 0), lam_over_mu=0.8),
                                _with(W.edge_crack(900, 200, 0, ny=610), wall_node=True)],
                         ids=lambda w: w.name)
def test_larger_lattices_bit_identical_to_one_step(wl):
    a = run_gpu(wl, 70, time_block=1)
    b = run_gpu(wl, 70)
    assert b["info"]["time_block"] > 1
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k], b[k]), k


def _run(wl, chunks, force=(0.0, 0.0), time_block=0):
    from paper_2208_04088_gb300 import _native as N
    d = N.desc_from_workload(wl, time_block=time_block)
    d.c.force[0], d.c.force[1] = force
    s = N.Solver(d)
    for c in chunks:
        s.step(c)
    s.sync()
    F = s.fields_host()
    s.close()
    return F


@pytest.mark.parametrize("lam", [1.0, 0.8], ids=["poisson", "nonpoisson"])
@pytest.mark.parametrize("force", [(0.0, 0.0), (3e-6, -2e-6)], ids=["", "force"])
def test_launch_of_two_kernels_bit_identical_to_one_step(force, lam):
    """Lattices with at least two interior tiles per SM: the tiles with boundary
    rules and the others go in kernels of their own, for full launches (replayed
    and single) and for every shorter one, where the next tile is not copied in
    ahead."""
    wl = _rules(1400, 1210, lam)
    a = _run(wl, [90], force, 1)
    b = _run(wl, [2, 3, 4, 5, 6, 7, 8, 16, 39], force)
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k], b[k]), k
    assert np.isfinite(a["u"]).all() and np.abs(a["u"]).max() > 0


@pytest.mark.parametrize("nx,ny", [(40, 33), (220, 150), (700, 500)])
def test_body_force_bit_identical_to_one_step(nx, ny):
    from paper_2208_04088_gb300 import _native as N
    wl, force = _rules(nx, ny), (-4e-6, 7e-6)
    a = _run(wl, [45], force, 1)
    b = _run(wl, [32, 13], force)
    free = N.desc_from_workload(wl)
    d = N.desc_from_workload(wl)
    d.c.force[0], d.c.force[1] = force
    batch = N.Batch([d, free])
    batch.step(45)
    batch.sync()
    c = batch.fields_host(0)
    batch.close()
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k], b[k]), k
        assert np.array_equal(a[k], c[k]), k


def test_batch_in_two_kernels_matches_instances_alone():
    """Enough interior tiles for a launch of two kernels; 37 steps leave launches
    of fewer than 8."""
    from paper_2208_04088_gb300 import _native as N
    wls = [W.hole_plate(1000, 900, 90.5, 0), _rules(640, 700), W.edge_crack(900, 200, 0, ny=600),
           W.hole_plate(96, 64, 9.0, 0)]
    b = N.Batch([N.desc_from_workload(w) for w in wls])
    b.step(37)
    b.sync()
    for k, w in enumerate(wls):
        ref = _run(w, [37], (0.0, 0.0), 1)
        got = b.fields_host(k)
        for q in ("u", "v", "sigma"):
            assert np.array_equal(got[q], ref[q]), (w.name, q)
    b.close()


@pytest.mark.parametrize("wl", [W.edge_crack(64, 16, 0), W.edge_crack(512, 128, 0, lam_over_mu=0.8),
                                W.edge_crack(1400, 300, 0)], ids=lambda w: f"{w.name}_{w.lam:.2g}")
def test_wait_limit_runs_out_cleanly(wl):
    """With a wait limit of 0 every tile gives up on its copy, waits it out and
    exits without storing; the host sees LBM_ERR_TIMEOUT, and after a reset with
    the limit back the handle runs on, bit-identical to one step per launch."""
    from paper_2208_04088_gb300 import _native as N
    s = N.Solver(N.desc_from_workload(wl))
    assert s.info()["time_block"] > 1
    N.lbm_set_wait_limit(s.h, 0)
    s.step(16)
    with pytest.raises(N.LbmError) as e:
        s.sync()
    assert e.value.status == N.LBM_ERR_TIMEOUT
    N.lbm_set_wait_limit(s.h, 10 ** 9)
    s.reset()
    s.step(43)
    s.sync()
    got = s.fields_host()
    s.close()
    ref = run_gpu(wl, 43, time_block=1)
    for k in ("u", "v", "sigma"):
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("lam", [1.0, 0.8], ids=["poisson", "nonpoisson"])
@pytest.mark.parametrize("nx,ny", [(150, 45), (300, 211)])
def test_fragmented_solid_bit_identical_to_one_step(nx, ny, lam):
    """Most nodes are boundary nodes (more than the larger tiles have slots
    for), cracks run through links, upstream nodes are missing."""
    bcs = [W.bc(W.DIRICHLET, (2e-4, -1.5e-4), W.RAMP, 20.0), W.bc(W.DIRICHLET, (-1e-4, 3e-4))]
    nt, cols = W.fragmented_solid(nx, ny, 7, void_frac=0.2, crack_frac=0.05, nbcs=len(bcs))
    a = run_gpu_tables(nt, cols, bcs, lam * W.MU, 45, time_block=1)
    b = run_gpu_tables(nt, cols, bcs, lam * W.MU, 45)
    assert b["info"]["time_block"] > 1
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k], b[k]), k
