"""Calls on a stream that is being captured into a graph. Calls that need
memory are refused in the capture modes that refuse cudaMalloc; where the mode
allows it the memory is the library's own, never the graph's. A box's stencils
reach the device during the call, not when the graph runs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

N, RC = 5000, 2.0
H = np.eye(3) * 20.0


def _points(seed):
    return torch.from_numpy(np.random.default_rng(seed).uniform(0, 20, size=(N, 3))).cuda()


def _count(P, cl):
    return P.cl_map(cl, "count")["count"].item()


@pytest.mark.parametrize("call", ["build", "grow", "cross"])
def test_refused_while_captured(cuda_ok, call):
    import paper_2202_06427_gb300 as P
    x, y = _points(1), _points(2)
    cl = P.cl_build(x, H, RC, 2)
    want, nbytes = _count(P, cl), P.cl_query(cl, "bytes")
    torch.cuda.synchronize()
    graph, code = torch.cuda.CUDAGraph(), 0
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin()
        try:
            if call == "build":
                P.cl_build(y, H, RC, 2)
            elif call == "grow":
                P.cl_update(cl, x, cutoff=1.0)
            else:
                P.cl_cross_count(cl, y)
        except P.CellMapError as e:
            code = e.code
        try:
            graph.capture_end()
        except RuntimeError:  # the refused call may have ended the capture
            pass
    assert code in (-5, -8)
    torch.cuda.synchronize()
    assert P.cl_query(cl, "bytes") == nbytes
    P.cl_update(cl, x)
    assert _count(P, cl) == want and _count(P, P.cl_build(x, H, RC, 2)) == want


def test_captured_update_to_another_box(cuda_ok):
    import paper_2202_06427_gb300 as P
    x, y = _points(1), _points(2)
    h = H.copy()
    h[1, 0], h[2, 1] = 1.5, -2.5
    want = [_count(P, P.cl_build(p, h, RC, 2)) for p in (x, y)]
    cl, held = P.cl_build(x, H, RC, 2), x.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin()
        P.cl_update(cl, held, h=h)
        graph.capture_end()
    other = P.cl_build(y, H * 1.3, RC, 3)  # the host's memory of the call is used again
    for p, w in zip((x, y), want):
        held.copy_(p)
        graph.replay()
        assert _count(P, cl) == w and _count(P, other) > 0
    near = P.cl_cross_count(cl, y)  # reads the stencil on the device
    assert near == P.cl_cross_count(P.cl_build(y, h, RC, 2), y)


def test_build_in_a_relaxed_capture(cuda_ok):
    """The list's memory is there at once; each replay builds it for the
    positions the tensor then holds."""
    import paper_2202_06427_gb300 as P
    x, y = _points(1), _points(2)
    want = [_count(P, P.cl_build(p, H, RC, 2)) for p in (x, y)]
    held = x.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin(capture_error_mode="relaxed")
        cl = P.cl_build(held, H, RC, 2)
        graph.capture_end()
    for p, w in zip((x, y, x), want + want[:1]):
        held.copy_(p)
        graph.replay()
        assert _count(P, cl) == w
    P.cl_free(cl)
    del graph
    assert _count(P, P.cl_build(x, H, RC, 2)) == want[0]
