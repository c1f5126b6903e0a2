"""The binning of sdot_power_spectrum: meshes on both sides of the 32 values of the last
index that a warp's first round covers, the mean |k| to the last fixed-point unit, and
transforms at the upper end of FP64 and beyond it.
"""
import math
from fractions import Fraction

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


def _k_units(M, nbins):
    """Per bin the sum over its modes of |n| in units of 2^-28, each rounded to the nearest
    (integer arithmetic throughout), and the mode counts."""
    f = np.fft.fftfreq(M, d=1.0 / M).astype(np.int64) ** 2
    d2 = np.bincount((f[:, None, None] + f[None, :, None] + f[None, None, :]).reshape(-1))
    units, cnt = [0] * nbins, [0] * nbins
    for v in np.flatnonzero(d2):
        v, m = int(v), int(d2[v])
        b = (math.isqrt(4 * v) + 1) // 2  # floor(sqrt(v) + 1/2)
        if 1 <= b <= nbins:
            r = (math.isqrt(v << 58) + 1) // 2  # sqrt(v) 2^28, rounded
            units[b - 1] += m * r
            cnt[b - 1] += m
    return units, cnt


@pytest.mark.parametrize("M", [31, 64, 200])
def test_mean_k_to_the_last_unit(M):
    # L = 2 pi: k is |n|. A bin's sum is below 2^52 units, so the one rounding of the mean
    # (the division by the count) moves it by less than half a unit of the sum
    nbins = 2 * M
    _, k, n = B.sdot_power_spectrum(np.ones((M, M, M)), 2.0 * math.pi, nbins)
    units, cnt = _k_units(M, nbins)
    np.testing.assert_array_equal(n, cnt)
    assert max(units) < 2 ** 52
    got = [round(Fraction(float(kb)) * c * 2 ** 28) for kb, c in zip(k, cnt)]
    assert got == units


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
