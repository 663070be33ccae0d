"""Levels of more than 32 cubes per axis, which the tile kernels serve, and the
grid transfers between such levels."""
import pytest
import torch

from synth import random_vector

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
