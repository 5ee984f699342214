"""Spectra of fields with a mean: the power of the corner mode (N/2, N/2, N/2), a shell
of its own, against an exact sum of the field with alternating signs, for sizes of the
library's own transforms and of cuFFT; and mode 0, the mean."""
import math

import numpy as np
import pytest

from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("N", [48, 100, 128, 160])  # the corner is alone in its shell
def test_corner_mode_of_a_field_with_a_mean(N, dtype):
    sigma, mean, kIR = 0.1, 0.5, 0.5
    npd = np.float32 if dtype == "f32" else np.float64
    f = (mean + sigma * np.random.default_rng(N).standard_normal((N, N, N))).astype(npd)
    with T.Lattice(N, kIR, 1, dtype) as lat:
        lat.set_state(f[None], np.zeros((1, N, N, N), npd))
        P = lat.spectrum(0, 0)[1]
    n = np.arange(N)
    sign = 1.0 - 2.0 * ((n[:, None, None] + n[None, :, None] + n) % 2)
    f = f.astype(np.float64)
    corner, total = math.fsum((f * sign).ravel()), math.fsum(f.ravel())
    V = (2.0 * math.pi / kIR) ** 3
    m = int(math.floor(math.sqrt(3.0) * N / 2.0 + 0.5))  # the corner's shell
    ref = V * (corner / N ** 3) ** 2
    # every row's sums of its even and odd columns round at about 2^-53 of N/2 values
    # of size sigma; over N^2 rows they add up at random: N^2/2 2^-53 sigma against the
    # mode; twice that for the power, four of these for the other passes' share
    tol = 8.0 * 2.0 ** -53 * (N ** 2 / 2.0) * sigma / abs(corner)
    assert abs(P[m] - ref) <= tol * ref, (P[m] / ref - 1.0, tol)
    assert abs(P[0] - V * (total / N ** 3) ** 2) <= 1e-14 * P[0]
