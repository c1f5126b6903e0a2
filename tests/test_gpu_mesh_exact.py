"""The mesh deposit against exact arithmetic: a lattice whose cells are boxes, strongly shrunk
and cut by a voxel edge on every axis. The density is a product of overlaps of intervals, in
fractions of the seeds' doubles.

Tolerance: a voxel edge in a cell's frame is (v h - y) / (s a) less the frame's origin: v h - y
rounds once (h is a power of two), the scale three times, the difference once, each to half
the cell; the facets of the cell round about as much. That is under 4 units in the last
place of the cell's width an axis, 12 for a piece, and its volume's sums a few more: 24 in all.
"""
from fractions import Fraction

import numpy as np
import pytest

from paper_2110_08868_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


def _overlaps(x, lam, M):
    """Fraction of cell i (the seeds x of a row, its facets half way between them, moved)
    that lies in voxel m of M, [i][m]."""
    n, s = len(x), 1 - Fraction(lam)
    xs = [Fraction(float(v)) for v in x]
    out = []
    for i in range(n):
        lo = (xs[i] + (xs[i - 1] if i else xs[-1] - 1)) / 2
        hi = (xs[i] + (xs[i + 1] if i + 1 < n else xs[0] + 1)) / 2
        lo, hi = xs[i] + s * (lo - xs[i]), xs[i] + s * (hi - xs[i])
        row = []
        for m in range(M):
            w = sum(max(Fraction(0), min(hi, Fraction(m + 1, M) + k) - max(lo, Fraction(m, M) + k))
                    for k in (-1, 0, 1))
            row.append(w / (hi - lo))
        out.append(row)
    return out


@pytest.mark.parametrize("lam", [0.5, 0.99])
def test_deposit_of_boxes_to_the_last_places(lam):
    n, M = 4, 8  # the sites lie on voxel edges, the seeds a little beside
    off = np.array([0.0007, -0.0004, 0.0003])
    y = np.ascontiguousarray(ics.lattice(n, 1.0) + off)
    with B.Solver(y, [1.0] * 3, precision="fp64") as s:
        s.laguerre(None)
        rho = s.mesh(lam, M)["rho"]
    ov = [_overlaps(y[:: n ** a][:n, a], lam, M) for a in range(3)]
    f = [[sum(o[i][m] for i in range(n)) for m in range(M)] for o in ov]
    scale = Fraction(M, n) ** 3
    tol = 24 * 2.0 ** -53 * float(scale)
    for z in range(M):
        for yy in range(M):
            for x in range(M):
                want = float(f[2][z] * f[1][yy] * f[0][x] * scale)
                assert abs(rho[z, yy, x] - want) <= tol, (z, yy, x, rho[z, yy, x], want)
