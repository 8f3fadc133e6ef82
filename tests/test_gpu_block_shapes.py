"""GPU: the block shapes of the one-step kernels, on both sides of the rules
that choose them, give the same bits."""
import numpy as np
import pytest

from paper_2208_04088_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _fields(desc, steps):
    from paper_2208_04088_gb300 import _native as N
    s = N.Solver(desc)
    s.step(steps)
    s.sync()
    F = s.fields_host()
    s.close()
    return F


def _same(a, b):
    for k in ("u", "v", "sigma"):
        assert np.array_equal(a[k].view(np.uint32), b[k].view(np.uint32)), k


def _plate(nx, ny):
    return W.hole_plate(nx, ny, min(nx, ny) / 6.3, 0)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny", [(511, 513), (512, 512), (512, 511), (515, 517), (1024, 1024), (1027, 1025)])
def test_one_lattice(nx, ny, storage):
    """Both ends of the rules for in place (512 columns, 2^18 nodes) and for two
    buffers (2^20 nodes, 16 bits beyond them and 1024 columns)."""
    from paper_2208_04088_gb300 import _native as N
    wl = _plate(nx, ny)
    two = _fields(N.desc_from_workload(wl, storage=storage, time_block=1), 37)
    _same(two, _fields(N.desc_from_workload(wl, storage=storage, in_place=True), 37))
