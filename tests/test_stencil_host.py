"""The neighbour-cell stencil of the host-side box preparation against the
definition: every integer offset whose two cells come nearer than the cutoff,
the distance minimised over the faces of the offset's parallelepiped. The
library decides most offsets by bounds and the rest by its exact solver; here
every offset is solved. No GPU needed."""
import itertools
import math

import numpy as np
import pytest


def _min_dist2(G, o):
    """min |sum_k d_k G_k|^2, d_k in [o_k - 1, o_k + 1], over all active sets."""
    dim = len(o)
    best = math.inf
    for pat in itertools.product((-1, 1, 0), repeat=dim):
        d = np.array([o[k] + pat[k] for k in range(dim)], dtype=float)
        free = [k for k in range(dim) if pat[k] == 0]
        if free:
            fixed = sum((d[k] * G[k] for k in range(dim) if k not in free), np.zeros(G.shape[1]))
            d[free] = np.linalg.lstsq(G[free].T, -fixed, rcond=None)[0]
            if any(abs(d[k] - o[k]) > 1 + 1e-12 for k in free):
                continue
        v = d @ G
        best = min(best, float(v @ v))
    return best


def _boxes():
    rng = np.random.default_rng(77)
    for dim in (2, 3):
        for lcell in (1, 2, 3, 4):
            yield np.eye(dim) * 10.0, 1.0 if dim == 2 else 2.5, lcell  # cells that fit exactly: touching corners
            yield np.diag(rng.uniform(8, 20, dim)), rng.uniform(1.0, 4.0), lcell
            h = np.diag(rng.uniform(8, 20, dim))
            for a in range(1, dim):
                for b in range(a):
                    h[a, b] = rng.uniform(-0.6, 0.6) * 8
            yield h, rng.uniform(1.0, 3.0), lcell
            yield h + rng.normal(scale=0.5, size=h.shape), rng.uniform(1.0, 3.0), lcell


@pytest.mark.parametrize("h,rc,lcell", list(_boxes()))
def test_stencil_holds_exactly_the_cells_within_the_cutoff(h, rc, lcell):
    import paper_2202_06427_gb300 as P
    info = P.cl_box_info(h, rc, lcell)
    n = np.array(info["grid"])
    w = np.array(info["widths"])
    G = h / n[:, None]
    reach = [math.ceil(rc * n[k] / w[k]) for k in range(len(n))]
    keep2 = rc * rc * (1 + 1e-9)
    near = sum(1 for o in itertools.product(*(range(-m, m + 1) for m in reach))
               if any(o) and _min_dist2(G, o) < keep2)
    assert info["stencil_full"] == 1 + near
    assert info["stencil_half"] == 1 + near // 2
