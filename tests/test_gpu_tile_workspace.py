"""GPU: the tables of the register tiles lie in the caller's workspace where it
has the part for strips (lambda = mu, at least 2^21 nodes)."""
import pytest

from paper_2208_04088_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HANDLES = 64


def _taken(desc):
    """Device bytes that 64 handles hold beside their (one, never stepped) workspace."""
    import torch
    from paper_2208_04088_gb300 import _native as N
    nbytes = N.lbm_workspace_size(desc)
    space = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    at = (space.data_ptr() + 255) // 256 * 256
    stream = torch.cuda.current_stream().cuda_stream
    N.lbm_destroy(N.lbm_create(desc, stream, at, nbytes))  # loads the kernels
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    held = [N.lbm_create(desc, stream, at, nbytes) for _ in range(HANDLES)]
    assert N.lbm_get_info(held[0])["time_block"] == (1 if desc.c.time_block == 1 else N.LBM_TIME_BLOCK)
    taken = free - torch.cuda.mem_get_info()[0]
    for h in held:
        N.lbm_destroy(h)
    return taken


def test_large_lattices_keep_their_tables_in_the_workspace():
    """Tables outside would be 1849 tiles of 32 bytes and 24 bytes for each of
    the 3 cut links of at least 4 x 2046 edge nodes: 0.6 MB and more a handle,
    beside the streams and events that a handle stepping singly holds too."""
    from paper_2208_04088_gb300 import _native as N
    wl = W.edge_crack(2048, 512, 0)
    _taken(N.desc_from_workload(wl, time_block=1))  # what the process keeps for later handles
    one = _taken(N.desc_from_workload(wl, time_block=1))
    tiles = _taken(N.desc_from_workload(wl))
    assert tiles - one < HANDLES * 300_000, (tiles, one)
