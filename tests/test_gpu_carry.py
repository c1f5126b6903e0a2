"""The carried pass (cells certified by their previous certificate, in a kernel of their
own) against the general pass: the same evaluations on a context with carrying off. Both do
the same FP32 arithmetic, so volumes and centroids may differ only by the order of their
FP64 sums (about 100 terms: 1e-13 relative) and facet coefficients not at all.
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
    if kind == "clumps":  # cells with many facets, far from their seeds, flagged for FP64
        y, _, _ = ics.zeldovich_box(n, 1.0, ics.spectrum_kinv, 0.3, 5)
        return np.ascontiguousarray(ics.add_clumps(y, 1.0, n, 2, 60, 0.05, 7)), [1.0] * 3
    if kind == "brick":   # a different grid along every axis
        rng = np.random.default_rng(n)
        L = np.array([1.0, 1.7, 0.6])
        return rng.uniform(0, 1, (n ** 3, 3)) * L, list(L)
    y, _, _ = ics.zeldovich_box(n, 1.0, ics.spectrum_kinv, 0.3, n)
    return y, [1.0] * 3


@pytest.mark.parametrize("kind,n", [("lattice", 5), ("lattice", 8), ("lattice", 31), ("brick", 13),
                                    ("brick", 17), ("clumps", 12)])
def test_carried_pass_equals_the_general_pass(kind, n):
    y, L = _box(kind, n)
    N = len(y)
    a2 = (np.prod(L) / N) ** (2.0 / 3.0)
    rng = np.random.default_rng(n)
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
                ev.append((g, info.carried, s.status()))
            out.append(ev)
    assert out[0][2][1] >= N // 3, "the carried pass did not run"
    for (g, _, st), (r, _, sr) in zip(*out):
        np.testing.assert_allclose(g["vol"], r["vol"], rtol=1e-12)
        dc = g["centroid"] - r["centroid"]
        dc -= np.array(L) * np.round(dc / L)
        assert np.abs(dc).max() <= 1e-12 * a2 ** 0.5
        np.testing.assert_array_equal(st, sr)
        assert abs(g["hess"] - r["hess"]).max() <= 1e-14 * abs(r["hess"]).max()
