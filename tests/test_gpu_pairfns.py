"""The mapped functions of the paper's examples, as C entry points built on the
functor hook: Code 5 (mass-weighted 1/r), Code 6/7 (Lennard-Jones energy and
forces), Code 10 (pairwise-velocity histogram), against the FP64 oracle's sums
over every pair-image."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity_util import BAND

pytestmark = pytest.mark.gpu

REGIMES = [(3, False, 3.0, 1), (3, True, 3.0, 2), (2, True, 4.0, 2), (3, True, 0.6, 2)]


def _set(dim, tric, rc_or_frac, seed):
    rng = np.random.default_rng(seed)
    if rc_or_frac < 1:  # small box: pairs with several images inside the cutoff
        h = np.eye(dim) * 9.0
        if tric:
            h[1, 0] = 2.0
        n_side = 9
        rc = rc_or_frac * oracle.geom_info(h, 1.0)["w"].min()
    else:
        L = 22.0 if dim == 3 else 50.0
        h = np.eye(dim) * L
        if tric:
            for a in range(1, dim):
                for b in range(a):
                    h[a, b] = rng.uniform(-0.25 * L, 0.25 * L)
        n_side = int(L)
        rc = rc_or_frac
    x = synth.jittered_fractional(h, n_side, n_side ** dim - 3, 0.4, seed + 1)
    x = x + rng.integers(-2, 3, size=x.shape).astype(np.float64) @ h
    return np.ascontiguousarray(x), h, rc


@pytest.mark.parametrize("dim,tric,rc,lcell", REGIMES)
def test_lj_energy_and_forces(cuda_ok, dim, tric, rc, lcell):
    import paper_2202_06427_gb300 as P
    x, h, rc = _set(dim, tric, rc, 300 + dim + 10 * tric + lcell)
    eps, sigma = 0.0442, 0.8
    ref = oracle.lj(x, h, rc, eps, sigma, band=BAND)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell)
    e, f = P.cl_map_lj(cl, eps, sigma)
    e0, _ = P.cl_map_lj(cl, eps, sigma, forces=False)
    slack = ref["band_abs_energy"]
    for got in (e.item(), e0.item()):
        assert abs(got - ref["energy"]) <= 1e-5 * ref["abs_energy"] + slack, (got, ref["energy"])
    fg = f.cpu().numpy().astype(np.float64)
    scale = np.abs(ref["forces"]).max()
    assert np.abs(fg - ref["forces"]).max() <= 1e-4 * scale + np.abs(ref["band_forces"]).max()


@pytest.mark.parametrize("dim,tric,rc,lcell", REGIMES)
def test_mass_potential(cuda_ok, dim, tric, rc, lcell):
    import paper_2202_06427_gb300 as P
    x, h, rc = _set(dim, tric, rc, 400 + dim + 10 * tric + lcell)
    m = np.random.default_rng(5).uniform(0.5, 2.0, size=x.shape[0]).astype(np.float32)
    ref = oracle.mass_potential(x, h, rc, m.astype(np.float64), band=BAND)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell)
    got = P.cl_map_mass(cl, torch.from_numpy(m).cuda()).item()
    assert abs(got - ref["value"]) <= 1e-5 * abs(ref["value"]) + ref["band"]


@pytest.mark.parametrize("dim,tric,rc,lcell", REGIMES)
def test_velocity_histogram(cuda_ok, dim, tric, rc, lcell):
    import paper_2202_06427_gb300 as P
    x, h, rc = _set(dim, tric, rc, 500 + dim + 10 * tric + lcell)
    v = np.random.default_rng(6).normal(size=x.shape).astype(np.float32)
    nbins = 10
    binstep = rc / 10.0
    ref = oracle.velocity_hist(x, h, rc, v.astype(np.float64), binstep, nbins, band=BAND)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell)
    counts, vsum = P.cl_map_velocity_hist(cl, torch.from_numpy(v).cuda(), binstep, nbins)
    c = counts.cpu().numpy()
    # a pair near a bin edge (or the cutoff) may land in its bin or a neighbour
    bc, bv = ref["band_counts"], ref["band_vsum"]
    near_c = bc + np.roll(bc, 1) + np.roll(bc, -1)
    near_v = bv + np.roll(bv, 1) + np.roll(bv, -1)
    assert np.all(c >= ref["counts"]) and np.all(c <= ref["counts"] + near_c), (c, ref["counts"])
    dv = vsum.cpu().numpy() - ref["vsum"]
    assert np.all(dv >= -1e-5 * ref["vsum"] - 1e-9) and np.all(dv <= 1e-5 * ref["vsum"] + near_v + 1e-9)


def test_pair_functions_reject_bad_arguments(cuda_ok):
    import paper_2202_06427_gb300 as P
    from paper_2202_06427_gb300 import CellMapError
    cl = P.cl_build(torch.zeros((4, 3), dtype=torch.float64, device="cuda") + 1.0, np.eye(3) * 10, 2.0, 2)
    with pytest.raises(CellMapError):
        P.cl_map_lj(cl, 1.0, 0.0)
    with pytest.raises(CellMapError):
        P.cl_map_velocity_hist(cl, torch.zeros((4, 3), device="cuda"), 0.5, 0)
    with pytest.raises(CellMapError):
        P.cl_map_velocity_hist(cl, torch.zeros((4, 3), device="cuda"), 0.5, 65)


@pytest.mark.parametrize("call", ["mass", "velocity"])
def test_failed_call_leaves_the_list_usable(cuda_ok, call):
    """A call that reports an error (here one that the calling thread had left
    pending) leaves nothing in the list's buffers: the forces are as before."""
    import ctypes
    import paper_2202_06427_gb300 as P
    from paper_2202_06427_gb300 import _lib
    lib = _lib.lib()
    n = 4000
    x = torch.from_numpy(np.random.default_rng(3).uniform(0, 20, size=(n, 3))).cuda()
    cl = P.cl_build(x, np.eye(3) * 20.0, 3.0, 1)
    want = P.cl_map(cl, "energy_forces_virial")["forces"]
    v = torch.ones((n, 3), dtype=torch.float32, device="cuda")
    out = torch.zeros(32, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    runtime = ctypes.CDLL("libcudart.so.13")
    assert runtime.cudaSetDevice(9999) != 0  # refused on the host; stays pending
    if call == "mass":
        code = lib.cl_map_mass(cl.handle, ptr(v), ptr(out), stream)
    else:
        code = lib.cl_map_velocity_hist(cl.handle, ptr(v), 0.3, 10, ptr(out), ptr(out[16:]), stream)
    assert code == -8 and runtime.cudaGetLastError() == 0
    got = P.cl_map(cl, "energy_forces_virial")["forces"]
    # the sums of a particle's forces come in another order from call to call
    assert torch.allclose(got, want, rtol=0, atol=1e-5 * want.abs().max().item())


@pytest.mark.parametrize("nbins", [1, 16, 17, 32, 33, 64])
def test_velocity_histogram_bins(cuda_ok, nbins):
    """The numbers of bins at which the sweep's blocks change their size."""
    import paper_2202_06427_gb300 as P
    x, h, rc = _set(3, True, 3.0, 640 + nbins)
    v = np.random.default_rng(7).normal(size=x.shape).astype(np.float32)
    binstep = rc / nbins
    ref = oracle.velocity_hist(x, h, rc, v.astype(np.float64), binstep, nbins, band=BAND)
    cl = P.cl_build(torch.from_numpy(x).cuda(), h, rc, 2)
    counts, vsum = P.cl_map_velocity_hist(cl, torch.from_numpy(v).cuda(), binstep, nbins)
    c = counts.cpu().numpy()
    bc, bv = ref["band_counts"], ref["band_vsum"]
    near_c = bc + np.roll(bc, 1) + np.roll(bc, -1)
    near_v = bv + np.roll(bv, 1) + np.roll(bv, -1)
    assert np.all(c >= ref["counts"]) and np.all(c <= ref["counts"] + near_c), (c, ref["counts"])
    dv = vsum.cpu().numpy() - ref["vsum"]
    assert np.all(dv >= -1e-5 * ref["vsum"] - 1e-9) and np.all(dv <= 1e-5 * ref["vsum"] + near_v + 1e-9)


def test_reciprocal_of_the_lennard_jones_sweep(cuda_ok, tmp_path):
    """Every float of a few binades, the ends of its range among them. Newton's
    step on an estimate w0 of relative error e0 <= 2^-23 leaves e0^2 and the
    rounding of 1 - v w0 (2^-24 e0), below 2^-45 together; the last fma rounds
    with 2^-24."""
    import ctypes
    import os
    import subprocess
    from paper_2202_06427_gb300 import build
    root = build.ROOT
    out = str(tmp_path / "librecip.so")
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-shared", "-cudart", "shared",
                   os.path.join(root, "tests", "recip_probe.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    worst = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for exponent in (-126, -20, -1, 0, 1, 7, 30, 125):
        first = (exponent + 127) << 23
        assert lib.recip_error(ctypes.c_uint(first), ctypes.c_uint(1 << 23), ctypes.c_void_p(worst.data_ptr())) == 0
    assert 0 < worst.cpu().view(torch.float64).item() <= 2.0 ** -24 * (1 + 2.0 ** -10)


@pytest.mark.parametrize("candidates", [79.5, 80.5])
@pytest.mark.parametrize("lcell", [1, 2])
def test_mass_potential_of_sparse_lists(cuda_ok, lcell, candidates):
    """Both sides of the 80 candidates per particle from which on the sum is the
    sweep's and not the functor's."""
    import paper_2202_06427_gb300 as P
    h = np.array([[26.0, 0, 0], [3.0, 25.0, 0], [-2.0, 4.0, 27.0]])
    rc = 2.5
    info = P.cl_box_info(h, rc, lcell)
    n = int(candidates * np.prod(info["grid"]) / info["stencil_half"])
    x = synth.jittered_fractional(h, int(np.ceil(n ** (1 / 3))), n, 0.4, 81)
    m = np.random.default_rng(9).uniform(0.5, 2.0, size=n).astype(np.float32)
    ref = oracle.mass_potential(x, h, rc, m.astype(np.float64), band=BAND)
    got = P.cl_map_mass(P.cl_build(torch.from_numpy(x).cuda(), h, rc, lcell), torch.from_numpy(m).cuda()).item()
    assert abs(got - ref["value"]) <= 1e-5 * abs(ref["value"]) + ref["band"]
