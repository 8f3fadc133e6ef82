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
@pytest.mark.parametrize("nx,ny", [(511, 513), (512, 512), (512, 511), (515, 517), (1024, 1024), (1027, 1025), (1501, 1399)])
def test_one_lattice(nx, ny, storage):
    """Both ends of the rules for in place (512 columns, 2^18 nodes) and for two
    buffers (2^20 nodes, 16 bits beyond 2^21 and 1024 columns)."""
    from paper_2208_04088_gb300 import _native as N
    wl = _plate(nx, ny)
    two = _fields(N.desc_from_workload(wl, storage=storage, time_block=1), 37)
    _same(two, _fields(N.desc_from_workload(wl, storage=storage, in_place=True), 37))


@pytest.mark.parametrize("form", ["f32", "bf16", "in_place"])
@pytest.mark.parametrize("count,nx,ny", [(2, 50, 41), (9, 100, 101), (25, 100, 101), (60, 100, 101), (260, 100, 101)])
def test_batch(count, nx, ny, form):
    """Batches stepped one step per launch, from less than a tile per SM to more
    than 144: one block per tile, per run of four, and the persistent grid."""
    from paper_2208_04088_gb300 import _native as N
    kw = dict(in_place=True) if form == "in_place" else dict(storage=form)
    wl = _plate(nx, ny)
    b = N.Batch([N.desc_from_workload(wl, **kw) for _ in range(count)])
    b.step(37)
    b.sync()
    alone = _fields(N.desc_from_workload(wl, time_block=0 if form == "in_place" else 1, **kw), 37)
    for i in {0, count // 2, count - 1}:
        _same(b.fields_host(i), alone)
    b.close()
