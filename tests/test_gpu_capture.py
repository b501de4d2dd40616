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


def _sweeps(P, cl):
    efv = P.cl_map(cl, "energy_forces_virial")
    return P.cl_map(cl, "energy")["energy"], efv["energy"], efv["forces"], P.cl_map(cl, "count")["count"]


def _same(got, want):
    for a, b in zip(got[:2], want[:2]):
        assert a.item() == pytest.approx(b.item(), rel=1e-6)
    assert (got[2] - want[2]).abs().max() <= 1e-5 * want[2].abs().max()
    assert got[3].item() == want[3].item()


def _sets():
    """One particle a cell or so, and the same number in an eighth of the box, on a
    jittered grid: cells of other sizes take other routes through the sweeps."""
    rng = np.random.default_rng(5)
    g = np.stack(np.meshgrid(*[np.arange(18)] * 3, indexing="ij"), -1).reshape(-1, 3)[:N]
    return [torch.from_numpy((g + 0.5 + rng.uniform(-0.2, 0.2, size=g.shape)) * s).cuda() for s in (20 / 18, 10 / 18)]


def test_sweeps_between_replays_of_an_update(cuda_ok):
    """A replayed update changes the cells without a call: the sweeps' work lists
    of the cells before must not be used."""
    import paper_2202_06427_gb300 as P
    sets = _sets()
    want = [_sweeps(P, P.cl_build(x, H, RC, 2)) for x in sets]
    held = sets[0].clone()
    cl = P.cl_build(held, H, RC, 2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin()
        P.cl_update(cl, held)
        graph.capture_end()
    for k in (0, 1, 0, 1):
        held.copy_(sets[k])
        graph.replay()
        _same(_sweeps(P, cl), want[k])


def test_replayed_sweeps_after_an_update(cuda_ok):
    """Sweeps captured on a list whose work lists were there, replayed after an
    update of the list."""
    import paper_2202_06427_gb300 as P
    sets = _sets()
    want = [_sweeps(P, P.cl_build(x, H, RC, 2)) for x in sets]
    cl = P.cl_build(sets[0], H, RC, 2)
    _sweeps(P, cl)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin()
        got = _sweeps(P, cl)
        graph.capture_end()
    for k in (1, 0, 1):
        P.cl_update(cl, sets[k])
        graph.replay()
        _same(got, want[k])
        _same(_sweeps(P, cl), want[k])
