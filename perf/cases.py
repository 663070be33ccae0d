"""The work that users of this library give it, for timing and comparison.

Every case calls the public Python API (`Context`, `Batch`, `StokesProblem` /
`stokes_velocity`) the way `bench.py`, the README and the tests do.  Fields
follow the library's own workloads: tanh spheres of jump 1e2..1e6, sums of
Gaussian log-viscosity bumps, a grid-unaligned tanh cube; sizes run from 8^3 to
256^3 velocity cubes, those whose coarsest grid is not 4^3 (N = 24, 48, ...)
among them.  Programs that iterate run on a stream of their own (`own_stream`),
as bench.py does; short scripts use the default stream, as the README does.

The mixed cycle computes in FP32 and hands its result over widened to FP64;
`run` returns it in FP32, which loses nothing.  The Krylov solves return the
solution and not the iteration count or the residual norm reached, which are
properties of one rounding history.
"""
import math

import numpy as np
import torch

import paper_2511_13109_gb300 as agca

NU = 10.0  # coarsening threshold of every workload
PREC = {"f64": agca.FP64, "mixed": agca.MIXED}
PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


def listed():
    return [
        # a unit-test-sized cycle: nothing but launches and latency
        dict(name="vcycle_f64_n4", op="vcycle", prec="f64", N=4, field="spheres", dr=1e4, own_stream=True),
        # the preconditioner of a medium solve in mixed precision (the 24-problem batch's smallest size)
        dict(name="vcycle_mixed_n32", op="vcycle", prec="mixed", N=32, field="spheres", dr=1e6, own_stream=True),
        # bench.py's headline workload, FP64 and mixed cycle: 51 M velocity unknowns
        dict(name="vcycle_f64_n128", op="vcycle", prec="f64", N=128, field="bumps", dr=1e6, own_stream=True),
        dict(name="vcycle_mixed_n128", op="vcycle", prec="mixed", N=128, field="bumps", dr=1e6, own_stream=True),
        # a caller's own multigrid on the level operators in FP32: finest and first coarse
        # operator, restriction, prolongation, on a grid of 97^3 vertices
        dict(name="levels_f32_n48", op="levels", prec="mixed", N=48, field="spheres", dr=1e6, own_stream=False),
        # the Stokes operator in FP64: true residuals of a caller's own Krylov method
        dict(name="stokes_f64_n64", op="stokes", prec="f64", N=64, field="spheres", dr=1e6, own_stream=False),
        # a new viscosity for an existing hierarchy (time stepping, inversion)
        dict(name="setup_mixed_n64", op="setup", prec="mixed", N=64, field="spheres", dr=1e6, own_stream=True),
        # uneven problems cycled together
        dict(name="batch_vcycle_mixed_12", op="batch", prec="mixed", N=64, count=12, field="sphere", dr=1e6, own_stream=True),
        # whole solves: MINRES in FP64 from a short script, mixed at 64^3 pressure cubes,
        # and the paper's FGMRES with BFBT
        dict(name="solve_f64_n16", op="solve", prec="f64", N=16, field="cube", dr=1e3, own_stream=False),
        dict(name="solve_mixed_n64", op="solve", prec="mixed", N=64, field="spheres", dr=1e2, own_stream=True),
        dict(name="fgmres_mixed_n32", op="fgmres", prec="mixed", N=32, field="cube", dr=1e4, own_stream=True),
        # one misfit gradient with respect to the element log-viscosity: forward and adjoint solve
        dict(name="adjoint_mixed_n24", op="adjoint", prec="mixed", N=24, field="spheres", dr=1e2, own_stream=True),
    ]


# N with a coarsest grid the library solves directly at moderate cost (2N / 2^k in 4..7)
SIZES = sorted({m << k for m in (2, 3) for k in range(8)} | {5, 7, 10, 14, 20, 28, 40, 56, 80, 112})
SPAN = {"vcycle": (4, 128), "levels": (4, 128), "stokes": (4, 128), "setup": (4, 64), "batch": (4, 64),
        "solve": (4, 32), "fgmres": (4, 32), "adjoint": (4, 24)}


def draw(rng):
    op = rng.choice(["vcycle", "vcycle", "vcycle", "vcycle", "levels", "levels", "stokes", "setup", "batch", "solve",
                     "fgmres", "adjoint"])
    lo, hi = SPAN[op]
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    N = min((n for n in SIZES if lo <= n <= hi), key=lambda n: abs(math.log(n / want)))
    c = dict(op=op, prec=rng.choice(["f64", "mixed"]), N=N, dr=float(10 ** rng.randint(2, 4 if op in ("solve", "fgmres", "adjoint") else 6)),
             field=rng.choice(["spheres", "bumps", "cube"]), own_stream=rng.random() < 0.7)
    if op in ("solve", "adjoint"):
        c["dr"] = 1e2 if op == "adjoint" else min(c["dr"], 1e3)
    if op == "batch":
        c.update(field="sphere", count=rng.randint(3, 16))
    if op == "fgmres":
        c.update(field="cube")
    return c


# ------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _field(case, N, seed):
    """Element means (at the centroids) of the viscosity and of the vertical
    forcing on the finest grid: eta (E,), f_z (E,)."""
    rng = np.random.default_rng([seed, N])
    dr, dev, n = float(case["dr"]), _device(), 2 * N
    kind = case["field"]
    if kind in ("spheres", "sphere"):
        cs = rng.uniform(0.2, 0.8, size=(8 if kind == "spheres" else 1, 3))
        rs = np.full(len(cs), 0.08) if kind == "spheres" else rng.uniform(0.05, 0.15, size=1)

        def fn(x, y, z):
            xi = torch.zeros_like(x)
            for (cx, cy, cz), r in zip(cs.tolist(), rs.tolist()):
                d = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2)
                xi = torch.maximum(xi, 0.5 * (1.0 - torch.tanh((d - r) / 0.01)))
            return dr ** -0.5 + (dr ** 0.5 - dr ** -0.5) * xi, -xi
    elif kind == "bumps":
        cs, amps, ws = rng.uniform(0, 1, size=(20, 3)), rng.uniform(-3, 3, size=20), rng.uniform(0.03, 0.15, size=20)
        top = 0.5 * math.log10(dr)

        def fn(x, y, z):
            lg = torch.zeros_like(x)
            for (cx, cy, cz), a, w in zip(cs.tolist(), amps.tolist(), ws.tolist()):
                lg += a * torch.exp(((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2) * (-0.5 / w ** 2))
            lg = lg.clamp(-top, top)
            return torch.pow(10.0, lg), -(lg + top) / (2 * top)
    else:  # a cube with tanh faces around an off-grid centre
        c = rng.uniform(0.42, 0.58, size=3).tolist()

        def fn(x, y, z):
            xi = torch.ones_like(x)
            for v, m in zip((x, y, z), c):
                xi = xi * 0.5 * (torch.tanh(20.0 * (v - m + 0.125)) - torch.tanh(20.0 * (v - m - 0.125)))
            return dr ** -0.5 + (dr ** 0.5 - dr ** -0.5) * xi, -xi
    # centroids of the six tetrahedra of a cube: coordinate p_k is (3 - k) / 4
    off = torch.tensor([[(3 - p.index(a)) / 4 for a in range(3)] for p in PERMS], dtype=torch.float64, device=dev)
    g = torch.arange(n, dtype=torch.float64, device=dev)
    eta = torch.empty(n, n, n, 6, dtype=torch.float64, device=dev)
    fz = torch.empty_like(eta)
    step = max(1, (1 << 24) // (6 * n * n))
    for k in range(0, n, step):
        z = (g[k:k + step, None, None, None] + off[:, 2]) / n
        y = (g[None, :, None, None] + off[:, 1]) / n
        x = (g[None, None, :, None] + off[:, 0]) / n
        eta[k:k + step], fz[k:k + step] = fn(*(t.expand(z.shape[0], n, n, 6) for t in (x, y, z)))
    return eta.reshape(-1), fz.reshape(-1)


def _forcing(fz):
    f = torch.zeros(3, fz.numel(), dtype=torch.float64, device=fz.device)
    f[2] = fz
    return f.reshape(-1)


def _noise(size, seed, k=0, dtype=torch.float64):
    g = torch.Generator(device=_device()).manual_seed(1000003 * seed + k)
    return torch.rand(size, generator=g, dtype=dtype, device=_device()) * 2 - 1


def _batch_sizes(case):
    N = int(case["N"])
    small = [n for n in SIZES if n <= N][-4:]
    return [small[(3 * i) % len(small)] for i in range(int(case["count"]))]


def _velocity_size(N):
    return 3 * (2 * N + 1) ** 3


def _inputs(case, seed):
    """The tensors of a case: everything that depends on the seed."""
    N, op = int(case["N"]), case["op"]
    if op == "batch":
        sizes = _batch_sizes(case)
        fields = [_field(case, n, 100 * seed + i)[0] for i, n in enumerate(sizes)]
        return {"sizes": sizes, "eta": fields, "r": [_noise(_velocity_size(n), seed, i) for i, n in enumerate(sizes)]}
    eta, fz = _field(case, N, seed)
    d = {"eta": eta}
    if op == "vcycle":
        d["r"] = _noise(_velocity_size(N), seed)
    elif op == "levels":
        t = torch.float32
        d.update(x=_noise(_velocity_size(N), seed, 0, t), xc=_noise(3 * (N + 1) ** 3, seed, 1, t))
    elif op == "stokes":
        d["x"] = _noise(_velocity_size(N) + (N + 1) ** 3, seed)
    elif op in ("solve", "fgmres"):
        d["f"] = _forcing(fz)
    elif op == "adjoint":
        d["f"] = _forcing(fz)
        d["theta"] = torch.log(eta)
        d["u_obs"] = 1e-3 * _noise(_velocity_size(N), seed)
    return d


def _tolerance(case):
    """Relative residual of the solves: below what the comparison of two
    solutions needs, above what FP64 rounding of K x allows."""
    return 1e-11 if int(case["N"]) <= 32 else 1e-10


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    s.stream = _stream() if case["own_stream"] else torch.cuda.default_stream(_device())
    with torch.cuda.stream(s.stream):
        s.d = d = _inputs(case, seed)
        op, N, prec = case["op"], int(case["N"]), PREC[case["prec"]]
        if op == "batch":
            s.batch = agca.Batch(d["sizes"], prec, device=_device(), stream=s.stream)
            s.batch.prepare(d["eta"], NU)
            s.z = [torch.empty_like(r) for r in d["r"]]
        elif op == "adjoint":
            s.problem = agca.StokesProblem(N, d["f"], None, prec, NU, rtol=_tolerance(case), device=_device(),
                                           rtol_adjoint=1e-10)
        else:
            s.ctx = agca.Context(N, None, prec, device=_device(), stream=s.stream)
            if op != "setup":
                s.ctx.prepare(d["eta"], NU)
            if op == "vcycle":
                s.z = torch.empty_like(d["r"])
            if op in ("solve", "fgmres"):
                s.b = s.ctx.load_vector(d["f"])
            if op == "stokes":
                s.y = torch.empty_like(d["x"])
            if op == "levels":
                s.y, s.yc = torch.empty_like(d["x"]), torch.empty_like(d["xc"])
    s.stream.synchronize()
    return s


_own = {}


def _stream():
    """One stream of the program's own for all that it does."""
    dev = _device().index
    if dev not in _own:
        _own[dev] = torch.cuda.Stream(device=dev)
    return _own[dev]


def run(s):
    op, d = s.case["op"], s.d
    with torch.cuda.stream(s.stream):
        if op == "vcycle":
            z = s.ctx.vcycle(d["r"], s.z)
            return z if s.case["prec"] == "f64" else z.to(torch.float32)
        if op == "batch":
            zs = s.batch.vcycle(d["r"], s.z)
            return zs if s.case["prec"] == "f64" else [z.to(torch.float32) for z in zs]
        if op == "levels":
            c, L = s.ctx, s.ctx.L
            dt = agca.F32 if s.case["prec"] == "mixed" else agca.F64
            x, xc, y, yc = (d["x"], d["xc"], s.y, s.yc) if dt == agca.F32 else (_wide(s, "x"), _wide(s, "xc"), None, None)
            return {"fine": c.apply(L, x, y, dtype=dt), "coarse": c.apply(L - 1, xc, yc, dtype=dt),
                    "restricted": c.restrict(L, x, dtype=dt), "corrected": c.prolong_add(L, xc, x.clone(), dtype=dt)}
        if op == "stokes":
            return s.ctx.stokes_apply(d["x"], s.y)
        if op == "setup":
            c = s.ctx
            c.prepare(d["eta"], NU)
            info = [c.level_info(l) for l in range(1, c.L + 1)]
            return {"flagged": [int(i.n_flag) for i in info], "lambda": [float(i.lambda_) for i in info[1:]],
                    "diagonal": c.level_data(c.L, agca.FIELD_DIAG), "coarse_diagonal": c.level_data(c.L - 1, agca.FIELD_DIAG),
                    "flags": c.level_data(c.L - 1, agca.FIELD_FLAGS), "pressure_mass": c.level_data(c.L - 1, agca.FIELD_PMASS),
                    "coarsest": c.level_data(1, agca.FIELD_COARSE)}
        if op == "solve":
            return s.ctx.solve(s.b, _tolerance(s.case), 20000)[0]
        if op == "fgmres":
            return s.ctx.solve_fgmres(s.b, _tolerance(s.case), 2000, restart=50, schur="bfbt", z_iters=30)[0]
        theta = d["theta"].detach().requires_grad_(True)
        u = agca.stokes_velocity(theta, s.problem)
        loss = 0.5 * torch.sum((u - d["u_obs"]) ** 2)
        loss.backward()
        return {"u": u.detach(), "gradient": theta.grad}


def _wide(s, k):
    if k + "64" not in s.d:
        s.d[k + "64"] = s.d[k].double()
    return s.d[k + "64"]


# --------------------------------------------------------------------- work
def _cycle_work(N, size):
    """One V(2,2) cycle: the residual in and the correction out in FP64, the
    element coefficients in the cycle's precision; the arithmetic of the four
    finest operator applications with their epilogues in edge form (99 flops a
    vertex on average), an eighth of it on each coarser level."""
    V, E = (2 * N + 1) ** 3, 6 * (2 * N) ** 3
    return 48.0 * V + size * E, 8 / 7 * 4 * 99.0 * V


def work(case):
    N, op = int(case["N"]), case["op"]
    V, Vp, E = (2 * N + 1) ** 3, (N + 1) ** 3, 6 * (2 * N) ** 3
    size = 8 if case["prec"] == "f64" else 4
    if op == "vcycle":
        b, f = _cycle_work(N, size)
    elif op == "batch":
        b, f = (sum(v) for v in zip(*(_cycle_work(n, size) for n in _batch_sizes(case))))
    elif op == "levels":  # x read and y, x + P e written; restricted; coefficients of two levels
        b, f = size * (9 * V + 12 * Vp + E + E / 8), 87.0 * (V + Vp) + 45 * Vp + 9 * V
    elif op == "stokes":  # [u; p] in, K [u; p] out, coefficients
        b, f = 48.0 * V + 16.0 * Vp + 8.0 * E, 200.0 * V
    elif op == "setup":  # the viscosity in, the data of the levels out; 21 power iterations a level
        b, f = 8 / 7 * (8.0 * E + 24.0 * V), 8 / 7 * 21 * 87.0 * V
    else:
        # Krylov solves: viscosity and right-hand side in, solution out; the arithmetic of about a
        # hundred iterations of a cycle and K z (the count depends on the field), twice for a gradient
        cf = _cycle_work(N, size)[1]
        b, f = 8.0 * E + 16.0 * (3 * V + Vp), (2 if op == "adjoint" else 1) * 100 * (cf + 250.0 * V)
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------- exact
# The same mathematics in FP64 with plain tensor operations: element matrices of the
# symmetric gradient on Kuhn tetrahedra (P1), Galerkin products of flagged elements,
# V(2,2) Chebyshev cycle, Stokes operator, MINRES.
def _corners(t):
    c, v = [(0, 0, 0)], [0, 0, 0]
    for a in PERMS[t]:
        v[a] = 1
        c.append(tuple(v))
    return c


def _element_matrix(t):
    """12 x 12 matrix of a type-t tetrahedron for eta = 1, h = 1, times 6 (entries component * 4 + vertex)."""
    X = np.ones((4, 4))
    X[:, 1:] = _corners(t)
    G = np.linalg.inv(X)[1:].T  # row a: gradient of barycentric function a
    K = np.einsum("ai,bi,cd->cadb", G, G, np.eye(3)) + np.einsum("ad,bc->cadb", G, G)
    return np.rint(K.reshape(12, 12))


def _children():
    """Per parent type: the 8 children (cube offset, type) in ascending element order and the values of the parent's barycentric functions at their vertices."""
    out = []
    for p in PERMS:
        kids = []
        for oz in range(2):
            for oy in range(2):
                for ox in range(2):
                    for t in range(6):
                        v = (np.array([ox, oy, oz]) + np.array(_corners(t))) / 2.0
                        s = v[:, p]
                        lam = np.stack([1 - s[:, 0], s[:, 0] - s[:, 1], s[:, 1] - s[:, 2], s[:, 2]], axis=1)
                        if lam.mean(axis=0).min() > 0:
                            kids.append(((ox, oy, oz), t, lam))
        out.append(kids)
    return out


class _Plain:
    def __init__(self, N, eta, nu=NU):
        dev = eta.device
        self.N, self.L, self.dev = N, agca_levels(N), dev
        self.n = {l: (2 * N) >> (self.L - l) for l in range(1, self.L + 1)}
        self.K = [torch.tensor(_element_matrix(t), device=dev) for t in range(6)]
        L, kids = self.L, _children()
        self.mean, self.flag, self.idx, self.gal = {L: eta}, {L: None}, {}, {}
        mx, mn = eta, eta
        for l in range(L - 1, 0, -1):
            n, nf = self.n[l], self.n[l + 1]
            g = torch.arange(n, device=dev)
            origin = (2 * g[None, None, :] + nf * (2 * g[None, :, None] + nf * 2 * g[:, None, None])).reshape(-1)
            ch = torch.stack([torch.stack([6 * (origin + o[0] + nf * (o[1] + nf * o[2])) + t for o, t, _ in kids[tp]], -1)
                              for tp in range(6)], 1).reshape(-1, 8)
            self.mean[l] = self.mean[l + 1][ch].mean(-1)
            mx, mn = mx[ch].amax(-1), mn[ch].amin(-1)
            self.flag[l] = mx > nu * mn
            e = torch.nonzero(self.flag[l]).reshape(-1)
            self.idx[l] = torch.full((6 * n ** 3,), -1, dtype=torch.int64, device=dev)
            self.idx[l][e] = torch.arange(e.numel(), device=dev)
            self.gal[l] = torch.zeros(e.numel(), 12, 12, dtype=torch.float64, device=dev)
            for tp in range(6):
                sel = torch.nonzero(e % 6 == tp).reshape(-1)
                if not sel.numel():
                    continue
                for k, (o, t, lam) in enumerate(kids[tp]):
                    P = torch.tensor(np.kron(np.eye(3), lam), device=dev)
                    c = ch[e[sel], k]
                    C = self.mean[l + 1][c][:, None, None] / (6.0 * nf) * self.K[t]
                    if l + 1 < L:
                        f = self.idx[l + 1][c]
                        C = torch.where((f >= 0)[:, None, None], self.gal[l + 1][f.clamp(min=0)] if self.gal[l + 1].numel() else C, C)
                    self.gal[l][sel] += P.T @ C @ P
        self.diag, self.lam = {}, {}
        for l in range(1, L + 1):
            self.diag[l] = self._diagonal(l)

    def mask(self, l, x):
        y = torch.zeros_like(x)
        y[:, 1:-1, 1:-1, 1:-1] = x[:, 1:-1, 1:-1, 1:-1]
        return y

    def _dca(self, l, t):
        c = self.mean[l].reshape(-1, 6)[:, t]
        if self.flag[l] is not None:
            c = torch.where(self.flag[l].reshape(-1, 6)[:, t], torch.zeros_like(c), c)
        n = self.n[l]
        return c.reshape(n, n, n) / (6.0 * n)

    def _vertices(self, l, e):
        n = self.n[l]
        cube, t = e // 6, e % 6
        i, j, k = cube % n, (cube // n) % n, cube // (n * n)
        cor = torch.tensor([_corners(t) for t in range(6)], device=self.dev)[t]  # (F, 4, 3)
        return (i[:, None] + cor[..., 0]) + (n + 1) * ((j[:, None] + cor[..., 1]) + (n + 1) * (k[:, None] + cor[..., 2]))

    def _diagonal(self, l):
        n = self.n[l]
        y = torch.zeros(3, n + 1, n + 1, n + 1, dtype=torch.float64, device=self.dev)
        for t in range(6):
            c, kd = self._dca(l, t), torch.diagonal(self.K[t]).reshape(3, 4)
            for a, (ox, oy, oz) in enumerate(_corners(t)):
                y[:, oz:oz + n, oy:oy + n, ox:ox + n] += kd[:, a, None, None, None] * c
        if l < self.L and self.gal[l].numel():
            e = torch.nonzero(self.flag[l]).reshape(-1)
            v = self._vertices(l, e)
            d = torch.diagonal(self.gal[l], dim1=1, dim2=2).reshape(-1, 3, 4)
            for c in range(3):
                y[c].view(-1).index_add_(0, v.reshape(-1), d[:, c].reshape(-1))
        y = self.mask(l, y)
        return y

    def apply(self, l, x):
        n = self.n[l]
        x = self.mask(l, x)
        y = torch.zeros_like(x)
        for t in range(6):
            cor = _corners(t)
            xe = torch.stack([x[:, oz:oz + n, oy:oy + n, ox:ox + n] for ox, oy, oz in cor], 1).reshape(12, -1)
            ye = ((self.K[t] @ xe).reshape(3, 4, n, n, n)) * self._dca(l, t)
            for a, (ox, oy, oz) in enumerate(cor):
                y[:, oz:oz + n, oy:oy + n, ox:ox + n] += ye[:, a]
        if l < self.L and self.gal[l].numel():
            e = torch.nonzero(self.flag[l]).reshape(-1)
            v = self._vertices(l, e)
            xe = x.reshape(3, -1)[:, v].permute(1, 0, 2).reshape(-1, 12, 1)
            ye = (self.gal[l] @ xe).reshape(-1, 3, 4)
            for c in range(3):
                y[c].view(-1).index_add_(0, v.reshape(-1), ye[:, c].reshape(-1))
        return self.mask(l, y)

    @staticmethod
    def prolong(e):
        m = e.shape[-1]
        f = torch.zeros(e.shape[0], 2 * m - 1, 2 * m - 1, 2 * m - 1, dtype=e.dtype, device=e.device)
        for d in range(8):
            dx, dy, dz = d & 1, (d >> 1) & 1, d >> 2
            f[:, dz::2, dy::2, dx::2] = 0.5 * (e[:, :m - dz, :m - dy, :m - dx] + e[:, dz:, dy:, dx:])
        return f

    @staticmethod
    def restrict(r):
        m = (r.shape[-1] + 1) // 2
        c = torch.zeros(r.shape[0], m, m, m, dtype=r.dtype, device=r.device)
        for d in range(8):
            dx, dy, dz = d & 1, (d >> 1) & 1, d >> 2
            s = 0.5 * r[:, dz::2, dy::2, dx::2]
            c[:, :m - dz, :m - dy, :m - dx] += s
            c[:, dz:, dy:, dx:] += s
        return c

    def smoother(self):
        """Largest eigenvalue estimates of D^-1 A (20 power iterations) and the coarsest matrix."""
        for l in range(2, self.L + 1):
            nv = self.n[l] + 1
            z = np.arange(1, 3 * nv ** 3 + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            u = ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
            v = self.mask(l, torch.from_numpy(2 * u - 1).to(self.dev).reshape(3, nv, nv, nv))
            inv = self._inverse(l)
            for _ in range(20):
                w = inv * self.apply(l, v)
                v = w / torch.linalg.vector_norm(w)
            self.lam[l] = float((v * self.apply(l, v)).sum() / (v * self.diag[l] * v).sum())
        self.coarsest = self._dense()

    def _inverse(self, l):
        d = self.diag[l]
        return torch.where(d > 0, 1.0 / torch.where(d > 0, d, torch.ones_like(d)), torch.zeros_like(d))

    def _dense(self):
        n = self.n[1]
        m = 3 * (n - 1) ** 3
        A = torch.zeros(m, m, dtype=torch.float64, device=self.dev)
        for q in range(m):
            x = torch.zeros(3, n + 1, n + 1, n + 1, dtype=torch.float64, device=self.dev)
            inner = torch.zeros(m, dtype=torch.float64, device=self.dev)
            inner[q] = 1.0
            x[:, 1:-1, 1:-1, 1:-1] = inner.reshape(3, n - 1, n - 1, n - 1)
            A[:, q] = self.apply(1, x)[:, 1:-1, 1:-1, 1:-1].reshape(-1)
        return A

    def chebyshev(self, l, b, x):
        lam, inv = self.lam[l], self._inverse(l)
        theta, delta = 0.6 * lam, 0.5 * lam
        d = inv * (b - (self.apply(l, x) if x is not None else 0.0)) / theta
        x = d if x is None else x + d
        rho = delta / theta
        rho1 = 1.0 / (2.0 * theta / delta - rho)
        return x + rho1 * rho * d + (2.0 * rho1 / delta) * (inv * (b - self.apply(l, x)))

    def vcycle(self, b, l=None):
        l = self.L if l is None else l
        if l == 1:
            x, m = torch.zeros_like(b), self.n[1] - 1
            x[:, 1:-1, 1:-1, 1:-1] = torch.linalg.solve(self.coarsest, b[:, 1:-1, 1:-1, 1:-1].reshape(-1)).reshape(3, m, m, m)
            return x
        x = self.chebyshev(l, b, None)
        r = b - self.apply(l, x)
        e = self.vcycle(self.mask(l - 1, self.restrict(self.mask(l, r))), l - 1)
        return self.chebyshev(l, b, x + self.mask(l, self.prolong(e)))

    # [u; p] with p on the coarser grid; B = -P^T B_f, (B_f u)_a = sum_T |T| / 4 div u
    def split(self, x):
        nv, m = 2 * self.N + 1, self.N + 1
        return x[:3 * nv ** 3].reshape(3, nv, nv, nv), x[3 * nv ** 3:].reshape(1, m, m, m)

    def stokes(self, x):
        u, p = self.split(x)
        n = 2 * self.N
        u, q = self.mask(self.L, u), self.prolong(p)[0]
        y, s = self.apply(self.L, u), torch.zeros_like(q)
        for t in range(6):
            X = np.ones((4, 4))
            X[:, 1:] = _corners(t)
            G = np.linalg.inv(X)[1:].T
            box = [(slice(oz, oz + n), slice(oy, oy + n), slice(ox, ox + n)) for ox, oy, oz in _corners(t)]
            qm = sum(q[b] for b in box) * (0.25 / (6.0 * n * n))
            div = sum(float(G[a, c]) * u[(c,) + box[a]] for a in range(4) for c in range(3) if G[a, c] != 0) * (0.25 / (6.0 * n * n))
            for a in range(4):
                s[box[a]] += div
                for c in range(3):
                    if G[a, c] != 0:
                        y[(c,) + box[a]] -= float(G[a, c]) * qm
        return torch.cat([self.mask(self.L, y).reshape(-1), -self.restrict(s[None]).reshape(-1)])

    def pressure_mass(self):
        N, n = self.N, 2 * self.N
        kids, inv = _children(), (1.0 / self.mean[self.L]).reshape(n, n, n, 6)
        m = torch.zeros(N + 1, N + 1, N + 1, dtype=torch.float64, device=self.dev)
        for t in range(6):
            w = sum(inv[o[2]::2, o[1]::2, o[0]::2, k] for o, k, _ in kids[t]) / 8 / (24.0 * N ** 3)
            for ox, oy, oz in _corners(t):
                m[oz:oz + N, oy:oy + N, ox:ox + N] += w
        return m

    def load(self, f):
        n = 2 * self.N
        f = f.reshape(3, n, n, n, 6)
        b = torch.zeros(3, n + 1, n + 1, n + 1, dtype=torch.float64, device=self.dev)
        for t in range(6):
            for ox, oy, oz in _corners(t):
                b[:, oz:oz + n, oy:oy + n, ox:ox + n] += f[..., t] / (24.0 * n ** 3)
        return torch.cat([self.mask(self.L, b).reshape(-1), torch.zeros((self.N + 1) ** 3, dtype=torch.float64, device=self.dev)])

    def solve(self, b):
        """MINRES with the block-diagonal preconditioner, repeated on the residual; pressure of mean zero."""
        mass = self.pressure_mass().reshape(-1)

        def pre(r):
            u, p = self.split(r)
            p = p.reshape(-1)
            z = (p - p.mean()) / mass
            return torch.cat([self.vcycle(self.mask(self.L, u)).reshape(-1), z - z.mean()])

        x = torch.zeros_like(b)
        for tol in (1e-8, 1e-6):
            x = x + self._minres(b - self.stokes(x), pre, tol)
        x[-mass.numel():] -= x[-mass.numel():].mean()
        return x

    def _minres(self, b, pre, tol):
        zero = torch.zeros_like(b)
        x, v0, v, w0, w = zero, zero, b, zero, zero
        z = pre(v)
        g = g0 = math.sqrt(float(z @ v))
        gp, eta, s0, s1, c0, c1 = 1.0, g, 0.0, 0.0, 1.0, 1.0
        for _ in range(1500):
            z = z / g
            k = self.stokes(z)
            d = float(k @ z)
            vn = k - (d / g) * v - (g / gp) * v0
            zn = pre(vn)
            gn = math.sqrt(max(0.0, float(zn @ vn)))
            a0, a2, a3 = c1 * d - c0 * s1 * g, s1 * d + c0 * c1 * g, s0 * g
            a1 = math.hypot(a0, gn)
            c, s = a0 / a1, gn / a1
            w0, w = w, (z - a3 * w0 - a2 * w) / a1
            x = x + c * eta * w
            eta = -s * eta
            if abs(eta) <= tol * g0 or gn == 0.0:
                break
            v0, v, z, gp, g = v, vn, zn, g, gn
            s0, s1, c0, c1 = s1, s, c1, c
        return x


def agca_levels(N):
    n, L = 2 * N, 1
    while n % 2 == 0 and n >= 8:
        n, L = n // 2, L + 1
    return L


def exact(case, seed):
    op, N = case["op"], int(case["N"])
    if op in ("solve", "fgmres", "adjoint") and N > 16:
        return None  # a plain Krylov solve takes minutes
    d = _inputs(case, seed)
    if op == "batch":
        return [_exact_cycle(n, eta, r) for n, eta, r in zip(d["sizes"], d["eta"], d["r"])]
    if op == "vcycle":
        return _exact_cycle(N, d["eta"], d["r"])
    p = _Plain(N, d["eta"])
    L, nv, m = p.L, 2 * N + 1, N + 1
    if op == "levels":
        x, xc = d["x"].double().reshape(3, nv, nv, nv), d["xc"].double().reshape(3, m, m, m)
        c = p.mask(L - 1, p.restrict(x))
        out = {"fine": p.apply(L, x), "coarse": p.apply(L - 1, xc), "restricted": c, "corrected": x + p.mask(L, p.prolong(xc))}
        return {k: v.reshape(-1) for k, v in out.items()}
    if op == "stokes":
        return p.stokes(d["x"])
    if op == "setup":
        p.smoother()
        return {"flagged": None, "lambda": [p.lam[l] for l in range(2, L + 1)], "diagonal": p.diag[L].reshape(-1),
                "coarse_diagonal": p.diag[L - 1].reshape(-1), "flags": None,
                "pressure_mass": p.pressure_mass().reshape(-1), "coarsest": p.coarsest.reshape(-1)}
    p.smoother()
    x = p.solve(p.load(d["f"]))
    if op != "adjoint":
        return x
    u = x[:3 * nv ** 3]
    rhs = p.mask(L, (u - d["u_obs"]).reshape(3, nv, nv, nv)).reshape(-1)
    lam, _ = p.split(p.solve(torch.cat([rhs, torch.zeros(m ** 3, dtype=torch.float64, device=x.device)])))
    U, n = p.mask(L, p.split(x)[0]), 2 * N
    lam, g = p.mask(L, lam), torch.empty(n, n, n, 6, dtype=torch.float64, device=x.device)
    for t in range(6):
        e = [torch.stack([w[:, oz:oz + n, oy:oy + n, ox:ox + n] for ox, oy, oz in _corners(t)], 1).reshape(12, -1) for w in (lam, U)]
        g[..., t] = -(e[0] * (p.K[t] @ e[1])).sum(0).reshape(n, n, n) / (6.0 * n) * d["eta"].reshape(n, n, n, 6)[..., t]
    return {"u": u, "gradient": g.reshape(-1)}


def _exact_cycle(N, eta, r):
    p = _Plain(N, eta)
    p.smoother()
    nv = 2 * N + 1
    return p.vcycle(p.mask(p.L, r.reshape(3, nv, nv, nv))).reshape(-1)
