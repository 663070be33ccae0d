"""The eight-lanes-per-vertex kernel of the small levels and the coarsest solve
by the explicit inverse, at the edges of their ranges: grids of 2 to 5 cubes
per axis, odd sizes, and the largest size (32 cubes); the first tiled sizes
(tiles cut in x and y, one and two tiled levels, nearly every coarse element
flagged) against the other precision on the same grid.  Tolerances as in
test_gpu_parity.py: 1e-12 (FP64) and 1e-5 (FP32) of the largest entry for an
apply, 1e-9 and 1e-4 for a cycle."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import agca as oagca
from oracle import stokes as ostokes
from synth import random_vector, sphere_sinkers

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2511_13109_gb300")
DEV = torch.device("cuda:0")


def _eta(N, seed):
    m = 6 * (2 * N) ** 3
    return np.exp(np.random.default_rng(seed).uniform(-2, 2, m) * np.log(10.0))


# (N, levels): finest / coarsest cubes per axis 4/2, 10/5, 12/3, 18/9 (1,536 coarsest unknowns)
@pytest.mark.parametrize("N,L", [(2, 2), (5, 2), (6, 3), (9, 2)])
@pytest.mark.parametrize("nu", [10.0, 1e9])  # nearly all elements flagged, none
def test_small_levels_match_oracle(N, L, nu):
    eta = _eta(N, N)
    H = oagca.Hierarchy(N, L, eta, nu)
    c64 = pkg.Context(N, L, pkg.FP64, device=DEV)
    c32 = pkg.Context(N, L, pkg.MIXED, device=DEV)
    for c in (c64, c32):
        c.prepare(torch.from_numpy(eta).to(DEV), nu)
    for l in range(1, L + 1):
        x = random_vector(3 * c64.V[l], 40 + l)  # boundary entries are not zero: they are ignored
        ref = H.A[l] @ (x * H.mask[l])
        big = np.abs(ref).max()
        xd = torch.from_numpy(x).to(DEV)
        for c in (c64, c32):  # FP64 with coefficient records, and from the element coefficients
            assert np.abs(c.apply(l, xd).cpu().numpy() - ref).max() <= 1e-12 * big, l
        x32 = x.astype(np.float32)
        ref = H.A[l] @ (x32.astype(np.float64) * H.mask[l])
        got = c32.apply(l, torch.from_numpy(x32).to(DEV), dtype=pkg.F32).cpu().numpy()
        assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max(), l
    r = random_vector(3 * c64.V[L], 50)
    ref = H.vcycle(r * H.mask[L])
    for c, tol in ((c64, 1e-9), (c32, 1e-4)):
        z = c.vcycle(torch.from_numpy(r).to(DEV)).cpu().numpy()
        assert np.abs(z - ref).max() <= tol * np.abs(ref).max()
        assert np.abs(z * (1 - H.mask[L])).max() == 0.0


# finest cubes per axis 32: the last point level; 36, 40, 48: tiles over point levels; 72: two tiled levels
@pytest.mark.parametrize("N", [16, 18, 20, 24, 36])
def test_point_kernel_meets_tile_kernel(N):
    eta = torch.from_numpy(_eta(N, N)).to(DEV)
    c64, c32 = (pkg.Context(N, None, p, device=DEV) for p in (pkg.FP64, pkg.MIXED))
    c64.prepare(eta, 10.0)
    c32.prepare(eta, 10.0)
    for l in (c64.L, c64.L - 1):
        x = torch.from_numpy(random_vector(3 * c64.V[l], l).astype(np.float32)).to(DEV)
        ref = c64.apply(l, x.double())
        big = float(ref.abs().max())
        assert float((c32.apply(l, x.double()) - ref).abs().max()) <= 1e-12 * big
        assert float((c32.apply(l, x, dtype=pkg.F32).double() - ref).abs().max()) <= 1e-5 * big
    r = torch.from_numpy(random_vector(3 * c64.V[c64.L], 7)).to(DEV)
    ref = c64.vcycle(r)
    assert float((c32.vcycle(r) - ref).abs().max()) <= 1e-4 * float(ref.abs().max())


# pressure grids of 2 to 9 cubes: no, one and several pressure vertices whose whole divergence stencil is interior
@pytest.mark.parametrize("N", [2, 3, 5, 9])
def test_stokes_coupling_matches_oracle(N):
    eta = _eta(N, 60 + N)
    S = ostokes.Stokes(oagca.Hierarchy(N, 2, eta, 10.0))
    x = random_vector(3 * (2 * N + 1) ** 3 + (N + 1) ** 3, N)
    xm = x.copy()
    xm[:S.nu_] *= S.mask  # boundary velocities are ignored
    ref = S.K(xm)
    for prec in (pkg.FP64, pkg.MIXED):
        c = pkg.Context(N, 2, prec, device=DEV)
        c.prepare(torch.from_numpy(eta).to(DEV), 10.0)
        y = c.stokes_apply(torch.from_numpy(x).to(DEV)).cpu().numpy()
        for part in (slice(None, S.nu_), slice(S.nu_, None)):
            assert np.abs(y[part] - ref[part]).max() <= 1e-12 * np.abs(ref[part]).max()


# tasks of the batched FP32 tiles travel as kernel parameters, 24 or 120 to a launch
@pytest.mark.parametrize("count", [25, 121])
def test_large_batch_equals_single(count):
    N = 18  # 36 cubes per axis: tiles on the finest level
    etas = [torch.from_numpy(_eta(N, s)).to(DEV) for s in (1, 2)]
    b = pkg.Batch([N] * count, pkg.MIXED, device=DEV)
    b.prepare([etas[i % 2] for i in range(count)], 10.0)
    r = [torch.from_numpy(random_vector(3 * (2 * N + 1) ** 3, 9 + i)).to(DEV) for i in range(2)]
    z = b.vcycle([r[i % 2] for i in range(count)])
    for i in range(2):
        c = pkg.Context(N, None, pkg.MIXED, device=DEV)
        c.prepare(etas[i], 10.0)
        ref = c.vcycle(r[i])
        for j in (i, count - 2 - (count - i) % 2, count - 1 - (count - 1 - i) % 2):
            assert torch.equal(z[j], ref), j


# a mixed context's finest coefficient records are the part of the workspace that FGMRES can do without;
# K z differs by rounding only, so both solves take the same iterations and meet the tolerance
@pytest.mark.parametrize("short, ok", [(0, True), (1, True), (2, False)])
def test_fgmres_workspace_without_records(short, ok):
    p = sphere_sinkers(18, 3, 0.15, 0.03, 1e2)  # 36 cubes per axis: past the point kernel
    c = pkg.Context(18, None, pkg.MIXED, device=DEV)
    c.prepare(torch.from_numpy(p.eta).to(DEV), 10.0)
    b = c.load_vector(torch.from_numpy(p.fbar.ravel()).to(DEV))
    x, it, rel = c.solve_fgmres(b, 1e-6, 400, 20)
    lib, sz = pkg.agca.lib(), ctypes.c_size_t()
    assert lib.agca_fgmres_workspace_size(c._h, 20, ctypes.byref(sz)) == 0
    records = (27 * 8 * c.V[c.L] + 255) // 256 * 256
    size = sz.value - records * min(short, 1) - 256 * (short == 2)
    work, y = torch.empty(size, dtype=torch.uint8, device=DEV), torch.empty_like(b)
    it2, rel2 = ctypes.c_int(), ctypes.c_double()
    st = lib.agca_solve_fgmres(c._h, b.data_ptr(), y.data_ptr(), 1e-6, 400, 20, 0, 30, work.data_ptr(), size,
                               ctypes.byref(it2), ctypes.byref(rel2))
    assert (st == 0) == ok
    if ok:
        assert it2.value == it and rel2.value <= 1e-6 and rel <= 1e-6
