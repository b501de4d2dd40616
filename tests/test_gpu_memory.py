"""The library's device memory: what is given back, and when."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

KEPT = 256 << 20  # freed memory that the library keeps for later calls
MARGIN = 64 << 20  # the driver maps memory in pieces of up to 32 MB; kernels loaded meanwhile


def _free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_freed_lists_go_back_to_the_device(cuda_ok):
    """cl_free returns a large list's memory, beyond what is kept, at once."""
    import paper_2202_06427_gb300 as P
    n = 16_000_000
    h = np.eye(3) * 1000.0
    x = torch.rand((n, 3), dtype=torch.float64, device="cuda") * 1000
    P.cl_free(P.cl_build(x[:1000].contiguous(), h, 100.0, 1))  # the pool and the kernels exist
    before = _free_bytes()
    cl = P.cl_build(x, h, 12.0, 1)
    assert P.cl_query(cl, "bytes") > KEPT + 2 * MARGIN
    P.cl_free(cl)
    left = before - torch.cuda.mem_get_info()[0]  # no synchronisation in between
    assert left <= KEPT + MARGIN


def test_two_set_workspace_goes_back_to_the_device(cuda_ok):
    """So does a two-set call its workspace (here 32 closest of 4M queries' lists)."""
    import paper_2202_06427_gb300 as P
    h = np.eye(3) * 1000.0
    x = torch.rand((10000, 3), dtype=torch.float64, device="cuda") * 1000
    y = torch.rand((4_000_000, 3), dtype=torch.float64, device="cuda") * 1000
    cl = P.cl_build(x, h, 12.0, 1)
    P.cl_cross_topk(cl, y[:100].contiguous(), 32)
    before = _free_bytes()
    P.cl_cross_topk(cl, y, 32)
    left = before - torch.cuda.mem_get_info()[0]
    assert left <= KEPT + MARGIN


def test_smaller_grid_gives_its_cells_back(cuda_ok):
    """A list updated to a grid of far fewer cells holds their memory no longer,
    and grows again; the pairs are those of a list built for the grid."""
    import paper_2202_06427_gb300 as P
    h = np.eye(3) * 1000.0
    x = torch.rand((20000, 3), dtype=torch.float64, device="cuda") * 1000
    cl = P.cl_build(x, h, 40.0, 2)
    small, want = P.cl_query(cl, "bytes"), P.cl_map(cl, "count")["count"].item()
    P.cl_update(cl, x, cutoff=3.0, lcell=1)
    large, fine = P.cl_query(cl, "bytes"), P.cl_map(cl, "count")["count"].item()
    assert large > small + (500 << 20)
    before = torch.cuda.mem_get_info()[0]
    P.cl_update(cl, x, cutoff=40.0, lcell=2)
    assert P.cl_query(cl, "bytes") == small
    assert torch.cuda.mem_get_info()[0] - before > large - small - KEPT - MARGIN
    assert P.cl_map(cl, "count")["count"].item() == want
    P.cl_update(cl, x, cutoff=3.0, lcell=1)
    assert P.cl_query(cl, "bytes") == large and P.cl_map(cl, "count")["count"].item() == fine
