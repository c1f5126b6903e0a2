"""The binning of sdot_power_spectrum: meshes on both sides of the 33 values of the last
index that a warp's first round covers, the mean |k| to the last fixed-point unit, and
transforms that overflow.
"""
import numpy as np
import pytest

import sdot_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402


# M / 2 + 1 values of the last index: one round (32), one more lane, two rounds, a remainder;
# one bin (rounds that end early), the default, every bin
@pytest.mark.parametrize("M", [62, 63, 64, 65, 100, 130])
def test_binning_rounds_match_the_oracle(M):
    rng = np.random.default_rng(M)
    L = 3.0
    rho = np.exp(0.3 * rng.standard_normal((M, M, M)))
    for nbins in (1, M // 2, 2 * M):
        P, k, n = B.sdot_power_spectrum(rho, L, nbins)
        Po, ko, no = O.power_spectrum(rho, L, nbins)
        np.testing.assert_array_equal(n, no)
        np.testing.assert_allclose(P, Po, rtol=1e-9, atol=0)
        np.testing.assert_allclose(k, ko, rtol=1e-9, atol=0)


def test_overflowing_transform_is_not_finite():
    # alternating planes of +-A whose transform overflows along the Nyquist wave number of x
    # (infinities and their differences) while the mean stays that of the plane of ones: the
    # bins holding those modes (from 8 on) report no finite power, the lower ones theirs
    M, A = 16, 4e306
    rho = np.broadcast_to(np.where(np.arange(M) % 2 == 0, A, -A), (M, M, M)).copy()
    rho[0] = 1.0
    P, _, n = B.sdot_power_spectrum(rho, 1.0, 12)
    assert np.all(n > 0)
    assert not np.isfinite(P[7:]).any(), P


def test_point_mass_near_the_largest_double():
    # |F_k|^2 = 1e308 for every mode: finite, but not the sum of the four modes (+-a, +-b, c).
    # P is L^3 in every bin (tolerance: the transform's rounding and the fixed point's)
    M, L = 16, 2.0
    rho = np.zeros((M, M, M))
    rho[3, 5, 7] = 1e154
    P, _, n = B.sdot_power_spectrum(rho, L, M)
    assert np.all(n[:13] > 0)
    np.testing.assert_allclose(P[:13], L ** 3, rtol=1e-9, atol=0)
