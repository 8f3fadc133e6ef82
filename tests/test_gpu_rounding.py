"""GPU: FP32 rounding against the FP64 oracle where a wave front shares it.

A front along a box edge gives every node of a row the same populations, so a
rounding that does not cancel in the momentum is shared by the row, kept from
step to step and added up by the displacement.  The bars are the errors of the
collision through all nine moments on the same runs (u and v; another
collision may be as far off, not further)."""
import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("load,shear,bar_u,bar_v", [
    (0.0009544448844578941, 6.796531688616956e-06, 1e-7, 2.8e-7),
    (0.00046157782128444856, 0.0002923661060027553, 1.3e-7, 3.3e-7)])
def test_front_along_the_edges(oracle_mod, load, shear, bar_u, bar_v):
    from paper_2208_04088_gb300 import _native as N
    wl = W.edge_crack(1100, 275, 400, load)
    wl.bcs[0] = W.bc(W.STRESS, (0.2 * shear, 0.1 * load, 0.0))
    wl.wall_node = True
    nt, links = oracle_mod.geometry(**wl.geometry_args())
    o = oracle_mod.Oracle(nt, links, wl.bcs, lam=wl.lam, mu=wl.mu, rho0=wl.rho0, tau=wl.tau,
                          wall_node=True)
    o.step(wl.steps)
    ref = o.fields()
    o.close()
    s = N.Solver(N.desc_from_workload(wl))
    s.step(wl.steps)
    s.sync()
    F = s.fields_host()
    s.close()
    mask = nt.astype(bool)
    for k, bar in (("u", bar_u), ("v", bar_v)):
        d, r = F[k][:, mask].astype(np.float64) - ref[k][:, mask], ref[k][:, mask]
        err = np.linalg.norm(d) / np.linalg.norm(r)
        assert err <= bar, (k, err)
