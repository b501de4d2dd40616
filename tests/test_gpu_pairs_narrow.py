"""Neighbour lists of boxes only a little wider than two cutoffs along an axis.
There the stencil reaches a cell from both sides (2 lcell + 1 > cells of the
axis), so one cell's staged neighbourhood holds two images of a particle: equal
indices, of which one at most lies within the cutoff. Lists against the oracle,
row by row, on grids of more than 64 particles per staging ball (a CTA per
cell) whose neighbourhoods fit the staging."""
import numpy as np
import pytest

import synth
from test_gpu_pairs import _check_against_oracle

pytestmark = pytest.mark.gpu

RC = 3.0

# faces' distances in cutoffs per axis, lcell, particles per axis of the lattice
CASES = {
    "cubic_2.001_l1": ((2.001,) * 3, 1, 9),
    "cubic_2.15_l1": ((2.15,) * 3, 1, 9),
    "cubic_2.90_l1": ((2.90,) * 3, 1, 10),
    "cubic_2.02_l2": ((2.02,) * 3, 2, 12),
    "cubic_2.26_l2": ((2.26,) * 3, 2, 12),
    "cubic_2.45_l2": ((2.45,) * 3, 2, 12),
    "cubic_2.10_l3": ((2.10,) * 3, 3, 12),
    "cubic_2.20_l4": ((2.20,) * 3, 4, 13),
    "outside_2.60_l2": ((2.60,) * 3, 2, 12),
    "slab_2.10_l2": ((6.3, 2.1, 5.2), 2, 17),
    "slab_2.40_l1": ((2.4, 5.1, 4.3), 1, 14),
    "flat_2.05_l2": ((2.05, 2.05), 2, 36),
    "flat_2.30_l3": ((2.30, 5.7), 3, 50),
    "flat_2.70_l1": ((2.70, 2.20), 1, 34),
}


def _box(widths, tric):
    """Rows of a box whose faces lie widths * RC apart."""
    d = len(widths)
    h = np.diag(np.array(widths) * RC)
    if tric:
        for a in range(1, d):
            for b in range(a):
                h[a, b] = (0.31, -0.22, 0.17)[a + b - 1] * h[b, b]
        w = 1.0 / np.linalg.norm(np.linalg.inv(h), axis=0)
        h *= (np.array(widths) * RC / w)[:, None]
        w = 1.0 / np.linalg.norm(np.linalg.inv(h), axis=0)
        assert np.allclose(w, np.array(widths) * RC)
    return h


def case_input(name, tric, order):
    widths, lcell, side = CASES[name]
    h = _box(widths, tric)
    x = synth.jittered_fractional(h, side, side ** len(widths) - 5, 0.4, 700 + side)
    if order == "random":
        x = x[np.random.default_rng(side).permutation(len(x))]
    return np.ascontiguousarray(x), h, lcell


@pytest.mark.parametrize("order", ["lattice", "random"])
@pytest.mark.parametrize("tric", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_list_of_a_narrow_box(cuda_ok, name, tric, order):
    import paper_2202_06427_gb300 as P
    x, h, lcell = case_input(name, tric, order)
    _check_against_oracle(P, x, h, RC, lcell)
