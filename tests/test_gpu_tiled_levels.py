"""Levels of more than 32 cubes per axis, which the tile kernels serve, and the
grid transfers between such levels."""
import pytest
import torch

from synth import random_vector, sphere_sinkers

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2511_13109_gb300")
DEV = torch.device("cuda:0")


# fine cubes per axis 18 to 256: coarse grids of 10 to 129 vertices a row, whole blocks and a remainder.
# The kernel adds d = 1 .. 7, +d before -d, and halves exactly, so plain sums in that order give the same bits.
@pytest.mark.parametrize("N, levels", [(36, (4, 3, 2)), (24, (4, 3)), (128, (7,))])
@pytest.mark.parametrize("dtype", [pkg.F64, pkg.F32])
def test_restriction_bit_exact(N, levels, dtype):
    c = pkg.Context(N, None, pkg.MIXED, device=DEV)
    td = torch.float64 if dtype == pkg.F64 else torch.float32
    for l in levels:
        n = 2 * N >> (c.L - l)
        r = torch.from_numpy(random_vector(3 * c.V[l], l)).to(DEV).to(td)
        got = c.restrict(l, r, dtype=dtype).view(3, n // 2 + 1, n // 2 + 1, n // 2 + 1)
        f = r.view(3, n + 1, n + 1, n + 1)

        def at(x, y, z):  # the interior coarse vertices, shifted on the fine grid
            return f[:, 2 + z:n - 1 + z:2, 2 + y:n - 1 + y:2, 2 + x:n - 1 + x:2]

        acc = torch.zeros_like(at(0, 0, 0))
        for d in range(1, 8):
            x, y, z = d & 1, (d >> 1) & 1, d >> 2
            acc = acc + at(x, y, z)
            acc = acc + at(-x, -y, -z)
        ref = torch.zeros_like(got)
        ref[:, 1:-1, 1:-1, 1:-1] = at(0, 0, 0) + 0.5 * acc
        assert torch.equal(got, ref), l


# A mixed context's coefficient records are the part of the FGMRES workspace that
# it can do without: a device that has no room for them still solves
@pytest.mark.parametrize("prec", [pkg.MIXED, pkg.FP64])
def test_fgmres_where_the_records_do_not_fit(prec, monkeypatch):
    p = sphere_sinkers(18, 3, 0.15, 0.03, 1e2)  # 36 cubes per axis: past the point kernel
    c = pkg.Context(18, None, prec, device=DEV)
    c.prepare(torch.from_numpy(p.eta).to(DEV), 10.0)
    b = c.load_vector(torch.from_numpy(p.fbar.ravel()).to(DEV))
    empty, sizes = torch.empty, []

    def no_room_for_the_first(*a, **k):
        if k.get("dtype") is torch.uint8:
            sizes.append(a[0])
            if len(sizes) == 1:
                raise torch.cuda.OutOfMemoryError("out of memory")
        return empty(*a, **k)

    monkeypatch.setattr(torch, "empty", no_room_for_the_first)
    if prec == pkg.FP64:  # nothing to leave out
        with pytest.raises(torch.cuda.OutOfMemoryError):
            c.solve_fgmres(b, 1e-6, 400, 20)
        return
    x, its, rel = c.solve_fgmres(b, 1e-6, 400, 20)
    assert rel <= 1e-6 and sizes[0] - sizes[1] >= 27 * 8 * c.V[c.L]


# levels of up to 32 cubes per axis run no tiles: the autotuner has nothing to time there
def test_autotuner_leaves_small_levels(tmp_path):
    cache = tmp_path / "tiles.txt"
    c = pkg.Context(16, None, pkg.MIXED, device=DEV)
    c.prepare(torch.from_numpy(sphere_sinkers(16, 3, 0.15, 0.03, 1e2).eta).to(DEV), 10.0)
    n = c.launch_count()
    assert set(c.autotune(2, str(cache)).values()) == {(8, 0)}
    assert c.launch_count() == n and cache.read_text() == ""
