"""The kNN lists of boxes under three grid cells thin along an axis, which the exact search
makes for every query (no 3^3 grid cells around it), with every list length it is built for,
against brute force with the same FP64 key. Integer results: bit-exact.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("L", [(1.0, 1.0, 0.03), (0.02, 1.0, 1.3), (1.0, 0.05, 0.9)])
@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 24, 25, 32, 33, 64])
def test_knn_of_a_thin_box(L, k):
    from test_gpu_knn import brute

    L = np.array(L)
    y = np.ascontiguousarray(np.random.default_rng(k).uniform(0, 1, (400, 3)) * L)
    want = brute(y, L, k)
    with B.Solver(y, list(L), k=k) as s:
        np.testing.assert_array_equal(s.knn(), want)
    if k <= B.SDOT_STATIC_MAX_K:
        nbr = torch.empty((len(y), k), dtype=torch.int32, device="cuda")
        rc = B.sdot_knn_static(torch.from_numpy(y).cuda(), list(L), k, nbr)
        if L[0] == 0.02:  # its grid has more cells than seeds, which the fixed array refuses
            assert rc == B.SDOT_ERR_ARG and "more grid cells than seeds" in B.sdot_last_error()
            return
        B.check(rc)
        np.testing.assert_array_equal(nbr.cpu().numpy(), want)
