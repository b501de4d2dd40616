"""The half-shell sweep's kinds of cells side by side: light cells (one warp),
fast-path cells, cells whose kept neighbourhood overflows the fast path, cells
of a batch's edge sizes (31-33, 64-65 particles), of more than 128 and of more
than 2,048. Every reduction against the oracle, and again on the same list,
whose work lists are kept (rules of parity_util)."""
import itertools

import numpy as np
import pytest
import torch

import oracle
from parity_util import BAND, TOL_GB, TOL_W, check_count, check_energy, check_forces, check_hist, check_matrix

pytestmark = pytest.mark.gpu


def _ball(rng, centre, radius, spacing, jitter):
    k = int(np.ceil(radius / spacing))
    g = np.stack(np.meshgrid(*[np.arange(-k, k + 1) * spacing] * 3, indexing="ij"), -1).reshape(-1, 3)
    g = g[np.linalg.norm(g, axis=1) <= radius]
    return centre + g + rng.uniform(-jitter, jitter, size=g.shape)


def _background(rng, h, spacing, centre, clear):
    n = max(1, int(np.abs(np.diag(h)).min() / spacing))
    s = np.stack(np.meshgrid(*[(np.arange(n) + 0.5) / n] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = s @ h + rng.uniform(-0.2, 0.2, size=s.shape) * spacing
    d = x - centre
    d -= np.round(d @ np.linalg.inv(h)) @ h
    return x[np.linalg.norm(d, axis=1) > clear]


CASES = {
    # light cells only: about three particles a cell, 40 in the half neighbourhood
    "light": dict(L=24.0, tric=True, rc=3.0, lcell=1, spacing=2.1, radius=0.0, fine=1.0),
    # a dense ball among light cells: neighbourhoods from a few to thousands, some
    # past the fast path's buffer although their raw count is below its limit
    "overflow": dict(L=24.0, tric=False, rc=3.0, lcell=2, spacing=1.6, radius=4.2, fine=0.42),
    # cells of about 32 and 64 particles, windowed by their dense neighbours
    "batches": dict(L=20.0, tric=True, rc=4.0, lcell=1, spacing=1.05, radius=4.5, fine=0.5),
    # a cell of more than 2,048 particles
    "huge": dict(L=16.0, tric=False, rc=4.0, lcell=1, spacing=1.5, radius=2.2, fine=0.26),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_kinds_of_cells(cuda_ok, name):
    import paper_2202_06427_gb300 as P
    c = CASES[name]
    rng = np.random.default_rng(len(name) + 31)
    h = np.eye(3) * c["L"]
    if c["tric"]:
        h[1, 0], h[2, 0], h[2, 1] = 3.1, -2.2, 1.7
    centre = np.array([0.375, 0.375, 0.375]) @ h  # the middle of a cell where the grid is four cells wide
    x = _background(rng, h, c["spacing"], centre, c["radius"] + 0.6 if c["radius"] else -1.0)
    if c["radius"]:
        x = np.vstack([x, _ball(rng, centre, c["radius"], c["fine"], 0.15 * c["fine"])])
    x = np.ascontiguousarray(x[rng.permutation(x.shape[0])])
    ref = oracle.pair_map(x, h, c["rc"], band=BAND, nbins=17)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, c["rc"], c["lcell"])
    g = torch.tensor([0.75], dtype=torch.float64, device="cuda")
    for _ in range(2):
        efv = P.cl_map(cl, "energy_forces_virial")
        check_energy(efv["energy"].item(), ref["energy"])
        check_forces(efv["forces"].cpu().numpy(), ref["forces"])
        check_matrix(efv["virial"].cpu().numpy(), ref["virial"], TOL_W)
        check_energy(P.cl_map(cl, "energy")["energy"].item(), ref["energy"])
        check_count(int(P.cl_map(cl, "count")["count"].item()), ref)
        check_hist(P.cl_map(cl, "hist", nbins=17)["hist"].cpu().numpy(), ref)
        gp, gb, _ = P.cl_backward(cl, g)
        check_forces(gp.cpu().numpy(), -0.75 * ref["forces"])
        check_matrix(gb.cpu().numpy(), 0.75 * ref["dedh"], TOL_GB)
    occupied = P.cl_query(cl, "max_occupancy")
    assert occupied > 2048 if name == "huge" else occupied <= 2048


@pytest.mark.parametrize("side", [19, 20, 22, 24])
@pytest.mark.parametrize("tric", [False, True])
def test_windowed_cells_in_no_order(cuda_ok, side, tric):
    """Uniform sets of 32 to 64 particles a cell on average, whose half
    neighbourhoods take two windows: the edges of the batches (32) and of the
    ordered cells (65), with and without a boundary in the stencil."""
    import paper_2202_06427_gb300 as P
    rng = np.random.default_rng(side)
    L, rc, lcell = 12.0, 4.0, 2
    h = np.eye(3) * L
    if tric:
        h[1, 0], h[2, 0], h[2, 1] = 1.1, -0.8, 0.7
    x = _background(rng, h, L / (side + 0.5), np.zeros(3), -1.0)
    assert len(x) == side ** 3
    x = np.ascontiguousarray(x[rng.permutation(len(x))])
    ref = oracle.pair_map(x, h, rc, band=BAND, nbins=17)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell)
    g = torch.tensor([0.75], dtype=torch.float64, device="cuda")
    for _ in range(2):
        efv = P.cl_map(cl, "energy_forces_virial")
        check_energy(efv["energy"].item(), ref["energy"])
        check_forces(efv["forces"].cpu().numpy(), ref["forces"])
        check_matrix(efv["virial"].cpu().numpy(), ref["virial"], TOL_W)
        check_energy(P.cl_map(cl, "energy")["energy"].item(), ref["energy"])
        check_count(int(P.cl_map(cl, "count")["count"].item()), ref)
        check_hist(P.cl_map(cl, "hist", nbins=17)["hist"].cpu().numpy(), ref)
        gp, gb, _ = P.cl_backward(cl, g)
        check_forces(gp.cpu().numpy(), -0.75 * ref["forces"])
        check_matrix(gb.cpu().numpy(), 0.75 * ref["dedh"], TOL_GB)


@pytest.mark.parametrize("lcell", [1, 2])
def test_clumps_beyond_each_others_cutoff(cuda_ok, lcell):
    """Clumps of 2 to 300 particles farther apart than the cutoff: a batch's own
    particles are all it is swept against (nothing listed), in the cells of one
    warp and, last batch by last batch, in the windowed ones."""
    import paper_2202_06427_gb300 as P
    rng = np.random.default_rng(8 + lcell)
    L, rc = 36.0, 3.0
    h = np.eye(3) * L
    h[2, 1] = 2.0
    sizes = [2, 3, 4, 5, 8, 31, 32, 33, 63, 64, 65, 128, 129, 160, 257, 300]
    sites = np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3) / 6 + 0.5 / 12
    x = []
    for k, s in enumerate(sites):
        g = np.stack(np.meshgrid(*[np.arange(-3, 4) * 0.2] * 3, indexing="ij"), -1).reshape(-1, 3)
        g = g[rng.permutation(len(g))[:sizes[k % len(sizes)]]]
        x.append(s @ h + g + rng.uniform(-0.05, 0.05, size=g.shape))
    x = np.vstack(x)
    x = np.ascontiguousarray(x[rng.permutation(len(x))])
    ref = oracle.pair_map(x, h, rc, band=BAND, nbins=17)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell)
    g = torch.tensor([0.75], dtype=torch.float64, device="cuda")
    for _ in range(2):
        efv = P.cl_map(cl, "energy_forces_virial")
        check_energy(efv["energy"].item(), ref["energy"])
        check_forces(efv["forces"].cpu().numpy(), ref["forces"])
        check_matrix(efv["virial"].cpu().numpy(), ref["virial"], TOL_W)
        gp, _, _ = P.cl_backward(cl, g)  # (no pair crosses the boundary: dE/dH is zero)
        check_forces(gp.cpu().numpy(), -0.75 * ref["forces"])


def _handed_over(x, h, rc, lcell):
    """Cells of at most 128 particles that the sweep lists for the fast path (the
    particles of the half neighbourhood, raw, within the share of the cells that
    lies in the staging ball) although those kept pass its buffer of 1,536."""
    hinv = np.linalg.inv(h)
    n = np.floor(lcell / np.linalg.norm(hinv, axis=0) / rc).astype(int)
    s = x @ hinv
    s -= np.floor(s)
    c = np.minimum((s * n).astype(int), n - 1)
    G = h / n[:, None]
    local = (s * n - c - 0.5) @ G
    assert np.allclose(h, np.diag(np.diag(h)))
    far = lambda o: sum((max(abs(v) - 1, 0) * G[k, k]) ** 2 for k, v in enumerate(o))
    off = [o for o in itertools.product(range(-lcell - 1, lcell + 2), repeat=3) if o[::-1] > (0, 0, 0) and far(o) < rc * rc]
    hd = 0.5 * np.linalg.norm(np.diag(G))
    cell = np.prod(np.diag(G))
    share = min(1.0, 0.5 * (4 / 3 * np.pi * (rc + hd) ** 3 - cell) / (cell * len(off)))
    cells = {}
    for i, k in enumerate(map(tuple, c)):
        cells.setdefault(k, []).append(i)
    found = 0
    for k, own in cells.items():
        near = [(j, o) for o in off for j in cells.get(tuple((np.array(k) + o) % n), [])]
        if len(own) > 128 or not 1536 < len(near) <= 1536 / share:
            continue
        j, o = np.array([v[0] for v in near]), np.array([v[1] for v in near])
        top = rc + np.linalg.norm(local[own], axis=1).max()
        found += np.linalg.norm(local[j] + o @ G, axis=1).__lt__(top).sum() > 1536
    return found


def test_cells_handed_over_by_the_sweep(cuda_ok):
    """Cells that the fast path finds too full while it stages them, and moves to
    the batches' list, which later calls on the same list take over: every
    reduction, the moving sweep first and last."""
    import paper_2202_06427_gb300 as P
    rng = np.random.default_rng(29)
    L, rc, lcell = 24.0, 6.0, 2
    h = np.eye(3) * L
    centre = np.array([10.5, 10.5, 10.5])  # the middle of a cell
    x = np.vstack([_background(rng, h, 1.2, centre, 1.6), _ball(rng, centre, 1.3, 0.215, 0.03)])
    x = np.ascontiguousarray(x[rng.permutation(x.shape[0])])
    assert len(x) >= 16 * 8 ** 3  # count and histogram staged as well
    assert _handed_over(x, h, rc, lcell) > 0
    ref = oracle.pair_map(x, h, rc, band=BAND, nbins=17)
    g = torch.tensor([0.75], dtype=torch.float64, device="cuda")

    def forces(cl):
        efv = P.cl_map(cl, "energy_forces_virial")
        check_energy(efv["energy"].item(), ref["energy"])
        check_forces(efv["forces"].cpu().numpy(), ref["forces"])
        check_matrix(efv["virial"].cpu().numpy(), ref["virial"], TOL_W)
        gp, gb, _ = P.cl_backward(cl, g)
        check_forces(gp.cpu().numpy(), -0.75 * ref["forces"])
        check_matrix(gb.cpu().numpy(), 0.75 * ref["dedh"], TOL_GB)

    def scalars(cl):
        check_energy(P.cl_map(cl, "energy")["energy"].item(), ref["energy"])
        check_count(int(P.cl_map(cl, "count")["count"].item()), ref)
        check_hist(P.cl_map(cl, "hist", nbins=17)["hist"].cpu().numpy(), ref)

    xd = torch.from_numpy(x).cuda()
    for order in ((forces, scalars, forces), (scalars, forces, scalars)):
        cl = P.cl_build(xd, h, rc, lcell)
        for part in order:
            part(cl)
