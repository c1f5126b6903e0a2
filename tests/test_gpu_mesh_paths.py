"""sdot_mesh where its paths differ: a cell with more facets than the small polytopes take, mesh
points on facets (the owners need a second pass), voxels much smaller and much larger than
the cells, and strongly shrunk cells. Against the oracle, tolerances as in test_gpu_mesh.
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


def _box(kind):
    if kind == "hub":
        from test_gpu_parity import hub_box

        return hub_box(n_sphere=40)[0]
    if kind == "lattice":
        return ics.lattice(6, 1.0)
    return ics.zeldovich_box(8, 1.0, ics.spectrum_kinv, 0.3, 3)[0]


@pytest.mark.parametrize("kind,M,lam", [("hub", 20, 0.3), ("lattice", 9, 0.0), ("lattice", 9, 0.5),
                                        ("box", 1, 0.2), ("box", 3, 0.9), ("box", 40, 0.0),
                                        ("box", 24, 0.97)])
def test_mesh_paths_match_the_oracle(kind, M, lam):
    y = _box(kind)
    psi = np.zeros(len(y))
    with B.Solver(y, [1.0] * 3, precision="fp64") as s:
        s.laguerre(psi)
        g = s.mesh(lam, M)
    rho = O.deposit(y, psi, 1.0, M, lam)
    np.testing.assert_allclose(g["rho"], rho, rtol=1e-9, atol=1e-9 * rho.max())
    phi, owner = O.potential_mesh(y, psi, 1.0, M)
    np.testing.assert_array_equal(g["phi"], phi)
    np.testing.assert_array_equal(g["owner"], owner)
