"""The kNN build (one warp a query, FP32 selection with exact ranking, exact search for what
does not fit) against brute force with the same FP64 key, where it can go wrong: grids of a
few cells an axis, ties, more seeds in a grid cell than the buffer holds, every range of k,
and boxes with a different grid along every axis. Integer results: bit-exact.
"""
import numpy as np
import pytest

from paper_2110_08868_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


def brute(y, L, k):
    out = np.empty((len(y), k), dtype=np.int32)
    for i in range(len(y)):
        d = y - y[i]
        d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
        key = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        key[i] = np.inf
        out[i] = np.lexsort((np.arange(len(y)), key))[:k]
    return out


def points(kind):
    rng = np.random.default_rng(12)
    if kind == "few":        # two grid cells an axis: every query takes the exact search
        return rng.uniform(0, 1, (30, 3)), np.ones(3)
    if kind == "lattice":    # shells of equal distances
        return ics.lattice(10, 1.0), np.ones(3)
    if kind == "clump":      # 500 seeds in one grid cell, far apart elsewhere
        c = 0.5 + 1e-3 * rng.standard_normal((500, 3))
        return np.concatenate([rng.uniform(0, 1, (700, 3)), c]), np.ones(3)
    L = np.array([1.0, 2.3, 0.4])
    return rng.uniform(0, 1, (1500, 3)) * L, L  # brick


@pytest.mark.parametrize("kind,k", [("few", 1), ("few", 29), ("lattice", 6), ("lattice", 26),
                                    ("lattice", 56), ("clump", 16), ("clump", 32), ("clump", 64),
                                    ("brick", 1), ("brick", 24), ("brick", 33), ("brick", 64)])
def test_knn_bit_exact(kind, k):
    y, L = points(kind)
    y = np.ascontiguousarray(y)
    with B.Solver(y, list(L), k=k) as s:
        np.testing.assert_array_equal(s.knn(), brute(y, L, k))
    if kind != "few" and k <= B.SDOT_STATIC_MAX_K:
        nbr = torch.empty((len(y), k), dtype=torch.int32, device="cuda")
        B.check(B.sdot_knn_static(torch.from_numpy(y).cuda(), list(L), k, nbr))
        np.testing.assert_array_equal(nbr.cpu().numpy(), brute(y, L, k))
