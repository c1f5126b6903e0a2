"""The mesh deposit where clips leave what is no polytope.

mesh_volume, which the deposit's masses are differences of, is compiled into a small program
with polytopes written by hand: it has to say that a vertex list is no polytope (NaN), since
any number would be taken for the volume of a piece. And boxes whose voxel planes lie on
facets, edges and vertices of the cells: the masses add up to the box's.
"""
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2110_08868_gb300 import build, ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


def test_volume_says_what_is_no_polytope(tmp_path):
    exe = str(tmp_path / "mesh_volume_test")
    r = subprocess.run([build.nvcc()] + build.ARCH + [
        "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
        os.path.join(HERE, "mesh_volume_test.cu"), "-o", exe], capture_output=True, text=True,
        timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    v = [float(x) for x in r.stdout.split()]
    assert len(v) == 8  # four cases, small and large polytopes
    for cube, off, missing, twice in (v[:4], v[4:]):
        # corners and their products are exact, the 24 terms' sum too
        assert cube == 8.0 and off == 8.0
        assert math.isnan(missing) and math.isnan(twice)


def _sites(kind, n):
    q = ics.lattice(n, 1.0)
    if kind == "cubic":
        return q
    off = np.array([[0, 0, 0], [.5, .5, .5]]) if kind == "bcc" else \
        np.array([[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]])
    return np.mod(np.concatenate([q + o / n for o in off]), 1.0)


# cells with more than three planes at a vertex (cubic, fcc) or facets along the axes (cubic,
# bcc: truncated octahedra), meshes and shrink factors that put voxel planes on them, and seeds
# off their sites by less and more than the tolerance of a clip (1e-13 of its terms)
@pytest.mark.parametrize("kind", ["cubic", "bcc", "fcc"])
@pytest.mark.parametrize("jitter", [0.0, 1e-14, 3e-13, 1e-12])
def test_density_of_nearly_degenerate_cells(kind, jitter):
    n = 4
    q = _sites(kind, n)
    y = np.mod(q + jitter * np.random.default_rng(n).standard_normal(q.shape), 1.0)
    y[y >= 1.0] = 0.0
    with B.Solver(np.ascontiguousarray(q), [1.0] * 3, precision="fp64") as s0, \
            B.Solver(np.ascontiguousarray(y), [1.0] * 3, precision="fp64") as s:
        s0.laguerre(None)
        s.laguerre(None)
        for lam in (0.0, 0.25, 1.0 / 3.0, 0.5, 0.75):
            for M in (n, 2 * n, 3 * n, 4 * n, 8 * n, 2 * n + 1):
                g = s.mesh(lam, M)
                rho = g["rho"]
                # pieces that overlap or leave a gap do so by the clip's tolerance
                assert abs(rho.mean() - 1.0) <= 1e-12, (lam, M, rho.mean() - 1.0)
                assert rho.min() >= 0.0
                # a facet moves by a few jitters, against a voxel of 1 / M and a contrast of
                # 1 / (1 - lam)^3; a plane that had to move aside, by 3e-11 a at most
                off = np.abs(rho - s0.mesh(lam, M)["rho"]).max()
                assert off <= 48 * (jitter + 3e-11 / n) * M / (1.0 - lam) ** 3, (lam, M, off)
