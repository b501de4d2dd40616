"""Rules that choose between two routes: the sizes on both sides of each rule
give the same results. Where the two routes run the same arithmetic in another
order of work (query order, key width) the outputs are compared bit for bit;
elsewhere against the oracle under the parity rules."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity_util import BAND, check_count, check_energy, check_forces, check_hist
from test_gpu_pairs import _check_against_oracle

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("dim,L,nb", [(3, 40.0, 16400), (2, 200.0, 10400)])
def test_query_order(cuda_ok, dim, L, nb):
    """About a set that passes the L2, many queries are taken in the order of
    their cells: the same lists, bit for bit, as in calls of at most 2,047."""
    import paper_2202_06427_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(31 + nb)
    n = (6 << 20) + 11
    h = np.eye(dim) * L
    h[1, 0] = 0.2 * L
    ht = torch.from_numpy(h).cuda()
    x = (3 * torch.rand((n, dim), generator=g, device="cuda", dtype=torch.float64) - 1) @ ht
    y = (3 * torch.rand((nb, dim), generator=g, device="cuda", dtype=torch.float64) - 1) @ ht
    cl = P.cl_build(x, h, 1.0, 1)
    assert 4 * nb >= P.cl_query(cl, "ncells")
    parts = [(s, y[s:s + 1999].contiguous()) for s in range(0, nb, 1999)]
    whole, lists = P.cl_cross_pairlist(cl, y), [P.cl_cross_pairlist(cl, p) for _, p in parts]
    assert P.cl_cross_count(cl, y) == sum(P.cl_cross_count(cl, p) for _, p in parts) == whole["a"].numel()
    assert torch.equal(whole["a"], torch.cat([q["a"] for q in lists]))
    assert torch.equal(whole["b"], torch.cat([q["b"] + s for q, (s, _) in zip(lists, parts)]))
    assert torch.equal(whole["d"], torch.cat([q["d"] for q in lists]))
    near, nears = P.cl_cross_knn(cl, y, 6), [P.cl_cross_knn(cl, p, 6) for _, p in parts]
    for k in range(2):
        assert torch.equal(near[k], torch.cat([q[k] for q in nears]))


def test_wide_keys(cuda_ok):
    """Lists over 2^22 particles sort segments by two-word keys. A cluster far
    from every other particle, numbered last among 4.2M, has the pairs (and
    distances, the grid being the same) it has in a list of its own."""
    import paper_2202_06427_gb300 as P
    m, a, rc = 162, 5.1, 5.0
    L = m * a
    h = np.eye(3) * L
    g = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * a
    rng = np.random.default_rng(77)
    u = rng.normal(size=(3500, 3))
    u *= (3.5 * rng.uniform(0, 1, size=(3500, 1)) ** (1 / 3)) / np.linalg.norm(u, axis=1, keepdims=True)
    u += 0.5 * L
    # no two sites and no site and cluster particle within the cutoff
    far = g[np.linalg.norm(g - 0.5 * L, axis=1) > 3.5 + rc + 0.1]
    assert len(far) > 1 << 22
    far = far[rng.permutation(len(far))]
    big, small = P.cl_build(_dev(np.vstack([far, u])), h, rc, 1), P.cl_build(_dev(u), h, rc, 1)
    want, got = P.cl_map(small, "pairlist"), P.cl_map(big, "pairlist")
    assert want["npairs"] == got["npairs"] > 1 << 20
    for k in ("i", "j"):
        assert torch.equal(got[k], want[k] + len(far))
    # a cell at the staging capacity may take the other route of the list here
    assert torch.allclose(got["d"], want["d"], rtol=0, atol=BAND * rc)
    y = _dev(u[::7] + rng.normal(size=u[::7].shape))
    want, got = P.cl_cross_pairlist(small, y), P.cl_cross_pairlist(big, y)
    # queries may reach the nearest sites
    mine = got["a"] >= len(far)
    assert torch.bincount(want["b"].long()).max() > 1024
    assert torch.equal(got["a"][mine], want["a"] + len(far)) and torch.equal(got["b"][mine], want["b"])
    assert torch.equal(got["d"][mine], want["d"])


@pytest.mark.parametrize("order", ["clumps", "rows", "random"])
def test_pairlist_numberings(cuda_ok, order):
    """The staged indices' spread over their range: tight clumps (compact
    blocks of 216 particles numbered together, 108 to a bucket, the radix
    sort), rows of the lattice, and random."""
    import paper_2202_06427_gb300 as P
    m, rc = 48, 3.0
    h = np.eye(3) * m
    rng = np.random.default_rng(91)
    s = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = s + 0.5 + rng.uniform(-0.3, 0.3, size=s.shape)
    if order == "clumps":
        block = ((s[:, 0] // 6) * 8 + s[:, 1] // 6) * 8 + s[:, 2] // 6
        x = x[np.argsort(rng.permutation(512)[block], kind="stable")]
    elif order == "random":
        x = x[rng.permutation(len(x))]
    _check_against_oracle(P, x, h, rc, 1)


@pytest.mark.parametrize("dim,lcell,rc,cluster", [(2, 1, 2.5, 0), (2, 3, 2.5, 2500), (2, 2, 2.5, 500), (3, 2, 1.4, 0),
                                                 (3, 1, 1.2, 700), (3, 3, 1.4, 2600)])
def test_pairlist_sparse_grids(cuda_ok, dim, lcell, rc, cluster):
    """At most 64 particles expected in a staging ball: a warp per cell, and a
    cluster whose cells take the larger staging (500, 700) or pass that too."""
    import paper_2202_06427_gb300 as P
    rng = np.random.default_rng(53 + cluster)
    L = 70.0 if dim == 2 else 18.0
    h = np.eye(dim) * L
    h[1, 0] = 0.1 * L
    x = synth.jittered_fractional(h, int(L), int(L) ** dim - 7, 0.4, 61)
    u = rng.normal(size=(cluster, dim))
    u *= (0.5 * rc * rng.uniform(0, 1, size=(cluster, 1)) ** (1 / dim)) / np.linalg.norm(u, axis=1, keepdims=True)
    x = np.vstack([x, u + 0.4 * L])
    _check_against_oracle(P, x[rng.permutation(len(x))], h, rc, lcell)


@pytest.mark.parametrize("ratio,lcell,tric", [(1.2, 1, False), (1.9, 1, True), (2.4, 2, True), (3.1, 1, True),
                                              (5.3, 3, False), (2.1, 4, False)])
def test_rows_of_small_2d_grids(cuda_ok, ratio, lcell, tric):
    """2D sweeps by rows of cells on grids down to one cell per axis, where a
    row's cells wrap onto each other."""
    import paper_2202_06427_gb300 as P
    rc = 4.0
    h = np.eye(2) * (ratio * rc)
    if tric:
        h[1, 0] = 0.15 * ratio * rc
        h *= ratio * rc / oracle.geom_info(h, rc)["w"].min()
    n_side = int(np.ceil(ratio * rc))
    x = synth.jittered_fractional(h, n_side, n_side ** 2, 0.3, 17)
    cl = P.cl_build(_dev(x), h, rc, lcell)
    ref = oracle.pair_map(x, h, rc, band=BAND, nbins=50)
    check_count(P.cl_map(cl, "count")["count"].item(), ref)
    check_hist(P.cl_map(cl, "hist", nbins=50)["hist"].cpu().numpy(), ref)
    out = P.cl_map(cl, "energy_forces_virial")
    check_energy(out["energy"].item(), ref["energy"])
    check_forces(out["forces"].cpu().numpy(), ref["forces"])


@pytest.mark.parametrize("occupancy", [1.5, 2.9, 3.1, 20.0])
@pytest.mark.parametrize("ratio,lcell,tric", [(1.2, 1, False), (1.9, 1, True), (2.4, 2, True), (3.1, 1, True),
                                              (9.3, 3, False), (6.1, 4, True)])
def test_2d_rows_and_cells(cuda_ok, ratio, lcell, tric, occupancy):
    """Both sides of the mean occupancy up to which 2D sweeps go by rows, on grids
    down to one cell per axis."""
    import paper_2202_06427_gb300 as P
    rc = 4.0
    h = np.eye(2) * (ratio * rc)
    if tric:
        h[1, 0] = 0.15 * ratio * rc
        h *= ratio * rc / oracle.geom_info(h, rc)["w"].min()
    cells = int(np.prod(P.cl_box_info(h, rc, lcell)["grid"]))
    n = max(2, int(occupancy * cells))
    side = int(np.ceil(np.sqrt(n)))
    x = synth.jittered_fractional(h, side, n, 0.3, 17)
    cl = P.cl_build(_dev(x), h, rc, lcell)
    ref = oracle.pair_map(x, h, rc, band=BAND, nbins=50)
    check_count(P.cl_map(cl, "count")["count"].item(), ref)
    check_hist(P.cl_map(cl, "hist", nbins=50)["hist"].cpu().numpy(), ref)
    if n >= 16:  # the relative rules are for sums over many pairs, not for two near the cutoff
        out = P.cl_map(cl, "energy_forces_virial")
        check_energy(out["energy"].item(), ref["energy"])
        check_forces(out["forces"].cpu().numpy(), ref["forces"])


@pytest.mark.parametrize("lcell,extra", [(3, -1), (3, 0), (4, -1), (4, 0)])
def test_pairlist_large_stencils(cuda_ok, lcell, extra):
    """Sparse grids of 300 and 600 stencil entries: a CTA per cell below 40
    particles per entry, a warp per cell from there on."""
    import paper_2202_06427_gb300 as P
    rc, L = 2.0, 60.0
    h = np.eye(3) * L
    h[1, 0], h[2, 1] = 4.0, -6.0
    n = 40 * P.cl_box_info(h, rc, lcell)["stencil_full"] + extra
    x = synth.jittered_fractional(h, int(np.ceil(n ** (1 / 3))), n, 0.5, 71)
    _check_against_oracle(P, x, h, rc, lcell)
