"""Cycles and solves whose finest, and first coarse, levels run the tile kernels
(more than 32 cubes per axis): against the oracle, against the same cycle put
together from single level operators, for every z-chunk, batched against alone,
and MINRES replayed from a graph against its direct launches.

Tolerances as in test_gpu_parity.py: 1e-12 (FP64) and 1e-5 (FP32) of the largest
entry for an apply, 1e-9 and 1e-4 for a cycle; equal bits where the operations
are the same."""
import numpy as np
import pytest
import torch

from oracle import agca as oagca
from oracle import fem
from synth import random_vector, sphere_sinkers

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2511_13109_gb300")
DEV = torch.device("cuda:0")
MODES = (1, 2, 3, 4)  # residual, first / later Chebyshev step, pre-smoothing step


def _random_eta(N, seed):
    return np.exp(np.random.default_rng(seed).uniform(-2, 2, 6 * (2 * N) ** 3) * np.log(10.0))


def _spheres(N, seed=77):
    return sphere_sinkers(N, 4, 0.11, 0.02, 1e4, seed=seed)


def _sharp(N, seed=78):  # jumps within an element's width: several times more flagged elements
    return sphere_sinkers(N, 4, 0.2, 0.002, 1e4, seed=seed)


def _ctx(N, prec, eta, stream=None):
    c = pkg.Context(N, None, prec, device=DEV, stream=stream)
    c.prepare(torch.from_numpy(np.ascontiguousarray(eta)).to(DEV), 10.0)
    return c


def _vec(n, seed):
    return torch.from_numpy(random_vector(n, seed)).to(DEV)


# 36 cubes per axis over 18 and 9: the finest level in tiles, nearly every coarse element flagged
def test_finest_tiles_match_oracle():
    N, L = 18, 3
    eta = _random_eta(N, 5)
    H = oagca.Hierarchy(N, L, eta, 10.0)
    c64, c32 = _ctx(N, pkg.FP64, eta), _ctx(N, pkg.MIXED, eta)
    assert c64.L == L
    x = random_vector(3 * c64.V[L], 3)
    ref = H.A[L] @ (x * H.mask[L])
    got = c64.apply(L, torch.from_numpy(x).to(DEV)).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    x32 = x.astype(np.float32)
    got = c32.apply(L, torch.from_numpy(x32).to(DEV), dtype=pkg.F32).cpu().numpy()
    assert np.abs(got - H.A[L] @ (x32.astype(np.float64) * H.mask[L])).max() <= 1e-5 * np.abs(ref).max()
    r = random_vector(3 * c64.V[L], 4)
    ref = H.vcycle(r * H.mask[L])
    for c, tol in ((c64, 1e-9), (c32, 1e-4)):
        z = c.vcycle(torch.from_numpy(r).to(DEV)).cpu().numpy()
        assert np.abs(z - ref).max() <= tol * np.abs(ref).max()
        assert np.abs(z * (1 - H.mask[L])).max() == 0.0


# the first coarse level of 72 cubes per axis: 36 cubes in tiles, with stored-Galerkin stencils
@pytest.mark.parametrize("field", [_spheres, _sharp])
def test_coarse_tiles_match_oracle(field):
    N, L = 36, 4
    p = field(N)
    H = oagca.Hierarchy(N, L, p.eta, 10.0, build_operators=False)
    m = H.mesh[L - 1]
    assert m.n == 36 and len(H.flist[L - 1]) > 0
    mask = fem.velocity_mask(m)
    A = fem.mask_matrix(fem.assemble(m, H.level_element_matrices(L - 1)), mask, mask)
    x32 = random_vector(3 * m.nv, 9).astype(np.float32)
    ref = A @ x32.astype(np.float64)
    big = np.abs(ref).max()
    x = torch.from_numpy(x32).to(DEV)
    c64, c32 = _ctx(N, pkg.FP64, p.eta), _ctx(N, pkg.MIXED, p.eta)
    for c in (c64, c32):  # FP64 with coefficient records, and from the element coefficients
        assert np.abs(c.apply(L - 1, x.double()).cpu().numpy() - ref).max() <= 1e-12 * big
    assert np.abs(c32.apply(L - 1, x, dtype=pkg.F32).cpu().numpy() - ref).max() <= 1e-5 * big


def _cycle_from_parts(c, r):
    """The V(2,2) cycle of an FP64 context from its level operators, diagonals
    and eigenvalue estimates, in plain FP64 vector operations."""
    inv, coarse = {}, None
    for l in range(1, c.L + 1):
        d = c.level_data(l, pkg.FIELD_DIAG)
        inv[l] = torch.where(d != 0, 1.0 / d, torch.zeros_like(d))
    inner = (inv[1] != 0).cpu().numpy()
    m = int(inner.sum())
    coarse = c.level_data(1, pkg.FIELD_COARSE).cpu().numpy().reshape(m, m)

    def smooth(l, b, x):
        lam = c.level_info(l).lambda_
        lo, hi = 0.1 * lam, 1.1 * lam
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        rho = delta / theta
        d = inv[l] * (b - c.apply(l, x)) / theta
        x = x + d
        rn = 1.0 / (2.0 * theta / delta - rho)
        return x + rn * rho * d + (2.0 * rn / delta) * (inv[l] * (b - c.apply(l, x)))

    def cycle(l, b):
        if l == 1:
            z = np.zeros(len(inner))
            z[inner] = np.linalg.solve(coarse, b.cpu().numpy()[inner])
            return torch.from_numpy(z).to(DEV)
        b = torch.where(inv[l] != 0, b, torch.zeros_like(b))
        x = smooth(l, b, torch.zeros_like(b))
        e = cycle(l - 1, c.restrict(l, b - c.apply(l, x)))
        return smooth(l, b, c.prolong_add(l, e, x))

    return cycle(c.L, r)


# finest cubes per axis 36, 40, 48, 72, 96: one and two tiled levels, tiles cut in x and y
@pytest.mark.parametrize("N", [18, 20, 24, 36, 48])
@pytest.mark.parametrize("field", [_spheres, _sharp])
def test_tiled_cycle_equals_its_parts(N, field):
    p = field(N)
    c64 = _ctx(N, pkg.FP64, p.eta)
    r = _vec(3 * c64.V[c64.L], 7)
    ref = _cycle_from_parts(c64, r)
    big = float(ref.abs().max())
    assert float((c64.vcycle(r) - ref).abs().max()) <= 1e-9 * big
    assert float((_ctx(N, pkg.MIXED, p.eta).vcycle(r) - ref).abs().max()) <= 1e-4 * big


@pytest.mark.parametrize("N, field", [(18, _spheres), (24, _spheres), (36, _spheres), (36, _sharp)])
@pytest.mark.parametrize("prec", [pkg.FP64, pkg.MIXED])
def test_tiled_cycle_independent_of_z_chunk(N, field, prec):
    c = _ctx(N, prec, field(N).eta)
    r = _vec(3 * c.V[c.L], 11)
    ref = c.vcycle(r).clone()
    dtype = pkg.F32 if prec == pkg.MIXED else pkg.F64
    xs = {l: _vec(3 * c.V[l], 20 + l).to(torch.float32 if prec == pkg.MIXED else torch.float64)
          for l in (c.L - 1, c.L)}
    ys = {l: c.apply(l, x, dtype=dtype).clone() for l, x in xs.items()}
    chunks = (1, 3, 7, 2 * N, 0)
    for i, _ in enumerate(chunks):
        for l in range(2, c.L + 1):
            for m in (0,) + MODES:  # a different chunk for every level and mode
                c.set_tile_config(l, m, 8, chunks[(i + l + m) % len(chunks)])
        assert torch.equal(c.vcycle(r), ref), i
        for l, x in xs.items():
            assert torch.equal(c.apply(l, x, dtype=dtype), ys[l]), (i, l)


@pytest.mark.parametrize("N", [24, 36])
@pytest.mark.parametrize("prec", [pkg.FP64, pkg.MIXED])
def test_tiled_autotune_round_trip(N, prec, tmp_path):
    cache = str(tmp_path / "tiles.txt")
    eta = _spheres(N).eta
    c = _ctx(N, prec, eta)
    r = _vec(3 * c.V[c.L], 5)
    ref = c.vcycle(r).clone()
    tuned = c.autotune(2, cache)
    assert set(tuned) == {(l, m) for l in range(2, c.L + 1) for m in MODES}
    assert torch.equal(c.vcycle(r), ref)
    c2 = _ctx(N, prec, eta)
    assert c2.autotune(2, cache) == tuned
    assert torch.equal(c2.vcycle(r), ref)


# uneven problems: point levels alone, tiles of several sizes, two tiled levels, with and without flagged elements
@pytest.mark.parametrize("prec", [pkg.FP64, pkg.MIXED])
@pytest.mark.parametrize("own_stream", [False, True])
def test_uneven_tiled_batch_equals_single(prec, own_stream):
    Ns = [36, 4, 18, 20, 24, 36]
    etas = [_spheres(N, 50 + i).eta for i, N in enumerate(Ns)]
    etas[2] = np.full(6 * 36 ** 3, 2.5)  # no element flagged
    etas[3] = _random_eta(20, 1)
    etas[5] = _sharp(36).eta
    s = torch.cuda.Stream(device=DEV) if own_stream else torch.cuda.current_stream(DEV)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        b = pkg.Batch(Ns, prec, device=DEV, stream=s)
        b.prepare([torch.from_numpy(e).to(DEV) for e in etas], 10.0)
        rs = [_vec(3 * c.V[c.L], 30 + i) for i, c in enumerate(b.contexts)]
        refs = [_ctx(N, prec, e, s).vcycle(r).clone() for N, e, r in zip(Ns, etas, rs)]
        zs = b.vcycle(rs)
        for i, (z, ref) in enumerate(zip(zs, refs)):
            assert torch.equal(z, ref), i
        zs = [r.clone() for r in rs]  # the result over the right-hand side
        for i, (z, ref) in enumerate(zip(b.vcycle(zs, zs), refs)):
            assert torch.equal(z, ref), i
    s.synchronize()


# Per-launch timing (profile_fine) switches graphs off, so that context launches directly.  36 cubes per axis and 8;
# an even and an odd number of iterations, and a solve to the end
@pytest.mark.parametrize("N", [4, 18])
@pytest.mark.parametrize("prec", [pkg.FP64, pkg.MIXED])
def test_minres_replay_equals_direct_launches(N, prec):
    p = _spheres(N)

    def solve(c, b, maxit):
        x = torch.zeros_like(b)
        try:
            return c.solve(b, 1e-8, maxit, x=x)
        except pkg.AgcaError as e:
            assert e.status == 4  # not converged: x holds the last iterate
            return x, None, None

    direct = _ctx(N, prec, p.eta)
    b = direct.load_vector(torch.from_numpy(p.fbar.ravel()).to(DEV))
    torch.cuda.synchronize()
    s = torch.cuda.Stream(device=DEV)
    for maxit in (2, 7, 5000):
        direct.profile_fine(True)
        ref = solve(direct, b, maxit)
        direct.profile_fine(False)
        replayed = _ctx(N, prec, p.eta)
        with torch.cuda.stream(s):
            own = _ctx(N, prec, p.eta, s)
            s.synchronize()
            for c in (replayed, own):
                for _ in range(2):  # capture, then the cached graph
                    got = solve(c, b, maxit)
                    torch.cuda.synchronize()
                    assert torch.equal(got[0], ref[0]) and got[1:] == ref[1:], maxit
