"""SU(2) step and measurement over the tile shapes and divisions of the lattice
among CTAs (one tile, ragged tiles, even division and z-chunks, fields staged
through shared memory or registers) and over the values FP32 widening
distinguishes, against the FP64 oracle."""
import numpy as np
import pytest

import oracle.su2 as Y
from paper_2607_24908_gb300 import tl as T
from paper_2607_24908_gb300.workloads import random_su2_links

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,N,steps", [("f64", 4, 3), ("f64", 7, 3), ("f64", 33, 3), ("f64", 50, 2), ("f64", 100, 1),
                                           ("f32", 4, 3), ("f32", 7, 3), ("f32", 33, 3), ("f32", 32, 3),
                                           ("f32", 96, 2), ("f32", 128, 1), ("f32", 150, 1)])
def test_step_over_tiles_matches_oracle(dtype, N, steps):
    tol = 1e-12 if dtype == "f64" else 1e-5  # as the parity tests of the step
    npd = np.float32 if dtype == "f32" else np.float64
    U0 = random_su2_links(N, seed=N, amp=0.6).astype(npd)
    E0 = (0.2 * np.random.default_rng(N).standard_normal((3, 3, N, N, N))).astype(npd)
    with T.SU2(N, dtype) as lat:
        lat.set_state(U0, E0)
        lat.step(steps, 0.05)
        U, E = lat.get_state()
    oU, oE = Y.step(U0.astype(np.float64), E0.astype(np.float64), 0.05, steps)
    assert np.max(np.abs(U - oU)) < tol
    assert np.max(np.abs(E - oE)) / np.max(np.abs(oE)) < tol


@pytest.mark.parametrize("dtype,fields", [("f64", "normal"), ("f32", "normal"), ("f32", "subnormal"), ("f32", "zero")])
def test_measure_of_any_stored_value(dtype, fields):
    """The measurement is FP64 arithmetic on the stored values: it agrees with the
    oracle on them to FP64 rounding, whatever mix of values the fields hold."""
    N = 9
    npd = np.float32 if dtype == "f32" else np.float64
    U = random_su2_links(N, seed=3, amp=0.6).astype(npd)
    E = np.random.default_rng(2).standard_normal((3, 3, N, N, N))
    if fields == "subnormal":
        E.reshape(-1)[::3] *= 1e-41
        E.reshape(-1)[1::3] = 0.0
    E = (E * (0.0 if fields == "zero" else 1.0)).astype(npd)
    with T.SU2(N, dtype) as lat:
        lat.set_state(U, E)
        m = lat.measure()
    U, E = U.astype(np.float64), E.astype(np.float64)
    G2 = np.sum(Y.gauss(U, E) ** 2, axis=0)
    for got, ref in zip(m, (Y.electric_energy(E), Y.plaquette_energy(U), np.sqrt(np.max(G2)), np.sqrt(np.mean(G2)))):
        assert abs(got - ref) <= 1e-13 * abs(ref), (m, ref)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_measure_shows_values_that_are_not_finite(bad):
    N = 8
    U = random_su2_links(N, seed=3, amp=0.6).astype(np.float32)
    E = np.ones((3, 3, N, N, N), np.float32)
    E[1, 2, 3, 4, 5] = bad
    with T.SU2(N, "f32") as lat:
        lat.set_state(U, E)
        assert not np.isfinite(lat.measure()[0])
