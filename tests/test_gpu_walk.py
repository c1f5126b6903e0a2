"""The security walk by a window of grid cells and its fallback to the pyramid, at the box
sizes where either can go wrong: grids too small for a pyramid (3 or 4 cells an axis),
windows as wide as the grid, windows that wrap, and a psi far above its surroundings
(whose window would hold too many cells). Every cell against the oracle.

Tolerances as in test_gpu_parity: FP64 1e-10 relative to a^3 and a; mixed 2e-5.
"""
import numpy as np
import pytest

import sdot_oracle as O
from paper_2110_08868_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 2e-5)])
@pytest.mark.parametrize("n,amp,peak", [(5, 0.03, 0.0), (6, 0.05, 0.0), (7, 0.1, 0.0),
                                        (9, 0.15, 0.0), (13, 0.2, 0.0), (13, 0.1, 1.2)])
def test_walk_window_edges(n, amp, peak, prec, tol):
    y, _, _ = ics.zeldovich_box(n, 1.0, ics.spectrum_kinv, 0.15, n)
    N, a = n ** 3, 1.0 / n
    nu = ics.uniform_masses(N, 1.0)
    rng = np.random.default_rng(n)
    psi = amp * a * a * rng.standard_normal(N)
    psi[rng.integers(N)] += peak * a * a
    s = B.Solver(y, [1.0] * 3, precision=prec)
    o = O.laguerre(y, psi, 1.0, nu, with_hessian=False)
    s.laguerre()  # the second diagram starts from the first one's facets
    for _ in range(2):
        g = s.laguerre(psi, allow_empty=True)
        np.testing.assert_allclose(g["vol"], o["vol"], rtol=0, atol=tol * a ** 3)
        ok = o["vol"] > 0
        dc = g["centroid"][ok] - o["centroid"][ok]
        dc -= np.round(dc)
        # the centroid of a nearly empty cell carries its volume's rounding
        assert np.max(np.abs(dc) * (o["vol"][ok, None] / a ** 3).clip(max=1)) <= tol * a
