"""The carried pass and the general pass give a cell the same bits: the same vertices, the
same sums in the same order (face by face on the same lanes), so what a call returns does not
depend on which pass took a cell. No tolerance: every value is compared for equality.
"""
import numpy as np
import pytest

from paper_2110_08868_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


def _box(kind, n):
    if kind == "clumps":  # cells with many facets, some flagged for the FP64 re-clip
        y, _, _ = ics.zeldovich_box(n, 1.0, ics.spectrum_kinv, 0.3, 5)
        return np.ascontiguousarray(ics.add_clumps(y, 1.0, n, 2, 60, 0.05, 7)), [1.0] * 3
    if kind == "brick":  # a different grid along every axis
        rng = np.random.default_rng(n)
        L = np.array([1.0, 1.7, 0.6])
        return rng.uniform(0, 1, (n ** 3, 3)) * L, list(L)
    y, _, _ = ics.zeldovich_box(n, 1.0, ics.spectrum_kinv, 0.3, n)
    return np.ascontiguousarray(y), [1.0] * 3


@pytest.mark.parametrize("kind,n", [("lattice", 5), ("lattice", 31), ("brick", 17), ("clumps", 12)])
def test_carried_pass_gives_the_general_pass_bits(kind, n):
    y, L = _box(kind, n)
    N = len(y)
    a2 = (np.prod(L) / N) ** (2.0 / 3.0)
    rng = np.random.default_rng(n + 1)
    psi = np.zeros(N)
    if kind == "clumps":
        with B.Solver(y, L, precision="fp64") as s:
            s.solve(1e-3)
            psi = s.psi()
    steps = [psi + 1e-4 * a2 * rng.standard_normal(N) for _ in range(3)]
    out, carried = [], []
    for carry in (1, 0):
        with B.Solver(y, L, precision="mixed", carry_certificates=carry) as s:
            ev = []
            for p in steps:
                g = s.laguerre(p, with_hessian=True)
                info = B.sdot_eval_info()
                B.check(B.sdot_last_eval(s.ctx, info))
                carried.append(info.carried)
                ev.append((g, s.status()))
            out.append(ev)
    assert carried[2] >= N // 3, "the carried pass did not run"
    assert carried[3:] == [0, 0, 0]
    for (g, st), (r, sr) in zip(*out):
        np.testing.assert_array_equal(st, sr)
        np.testing.assert_array_equal(g["vol"], r["vol"])
        np.testing.assert_array_equal(g["centroid"], r["centroid"])
        for part in ("indptr", "indices", "data"):
            np.testing.assert_array_equal(getattr(g["hess"], part), getattr(r["hess"], part))
