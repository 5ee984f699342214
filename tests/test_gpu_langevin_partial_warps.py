"""Langevin steps whose warps are partly filled: rows of 5, 7, 11 and 25 threads,
tiles cut by the end of a row or by the last row of the lattice."""
import numpy as np
import pytest

import oracle as o
from paper_2607_24908_gb300 import tl as T
from paper_2607_24908_gb300.workloads import white_noise_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-12), ("f32", 1e-5)])  # as the parity test of the step
@pytest.mark.parametrize("N", [8, 12, 20, 28, 44, 100, 132])
def test_partly_filled_warps_match_oracle(N, dtype, tol):
    npd = np.float32 if dtype == "f32" else np.float64
    kIR = 4.0 * np.pi / N  # dx = 1/2: the step is stable at every N
    phi0 = white_noise_state(N, 1, seed=N, phi0=(0.5,), sigma_phi=0.2)[0][0].astype(npd)
    with T.Lattice(N, kIR, 1, dtype) as lat:
        lat.set_state(phi0[None], np.zeros((1, N, N, N), npd))
        lat.langevin(6, 0.01, 1.0, 0.5, 1.0, 77)
        got = lat.get(0, 0)
    ref = o.langevin_run(N, kIR, phi0.astype(np.float64), 0.01, 6, 1.0, 0.5, 1.0, 77)
    assert np.max(np.abs(got - ref)) / np.max(np.abs(ref)) < tol
