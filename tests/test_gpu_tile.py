"""GPU: register-tile stepping, the default of most lattices (several steps per
launch, lbm_tile.cu).  Per node it performs the one-step arithmetic, so its
fields must be bit-identical to time_block = 1 for every tile shape, at the
edges of tiles and lattices, and for any split of a run into calls (a launch
carries any number of steps up to LBM_TIME_BLOCK)."""
import dataclasses

import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

from helpers import run_gpu

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
