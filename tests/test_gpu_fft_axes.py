"""The library's own transforms at every radix split (2^m, 3 2^m, 5 2^m; one to
three exchanges, 2 to 64 threads a line) and the sizes next to the rule that
chooses them: spectra and initial fields against the oracle, waves of known
power, and at the larger sizes a field of known modulus drawn and measured."""
import numpy as np
import pytest

import oracle as o
from paper_2607_24908_gb300 import tl as T
from paper_2607_24908_gb300.workloads import white_noise_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [60, 64, 80, 96, 128, 160, 192])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_spectrum_matches_oracle(N, dtype):
    npd = np.float32 if dtype == "f32" else np.float64
    phi, pi = white_noise_state(N, 1, seed=N, phi0=(0.5,), sigma_phi=0.1, sigma_pi=0.2)
    phi, pi = phi.astype(npd), pi.astype(npd)
    p = o.Params(N=N, nf=1, kIR=0.3)
    with T.Lattice(N, p.kIR, 1, dtype) as lat:
        lat.set_state(phi, pi)
        k, P, c = lat.spectrum(0, 0)
    ok, oP, oc = o.spectrum(p, phi[0].astype(np.float64))
    assert np.array_equal(c, oc) and c.sum() == N ** 3
    # |F|^2 to FFT rounding of the largest mode (the mean): 1e-14 of its amplitude, twice
    # that relative to the shell's own, and 1e-12 of the shell's power
    top = np.sqrt(np.max(oP))
    assert np.all(np.abs(P - oP) <= 1e-12 * oP + 2e-14 * top * np.sqrt(oP) + (1e-14 * top) ** 2)


@pytest.mark.parametrize("N", [64, 80, 96, 160])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_initial_fields_match_oracle(N, dtype):
    p = o.Params(N=N, nf=1, kIR=0.2, expanding=True, alpha=1.0, lam=1.0, q=0.0)
    spec = o.InitSpec(A=1e-8, meff2=(3.0, 0, 0), phi0=(1.0, 0.0, 0), fluct_pi=True, fixed_modulus=False)
    ophi, opi, _, _ = o.init_fluctuations(p, 5, spec)
    with T.Lattice(N, p.kIR, 1, dtype, True, 1.0, 1.0, 1.0) as lat:
        lat.set_potential(p.lam, p.q, (0, 0, 0))
        lat.init_fluctuations(5, A=1e-8, meff2=(3.0, 0, 0), phi0=(1.0, 0, 0), fluct_pi=True)
        phi, pi = lat.get_all()
    ulp = 2.0 ** -52 if dtype == "f64" else 2.0 ** -23
    # the fluctuation to 1e-12 of its size, plus roundings of the stored value
    for got, ref, mean in ((phi[0], ophi[0], 1.0), (pi[0], opi[0], 0.0)):
        size = np.max(np.abs(ref - mean))
        assert np.max(np.abs(got - ref)) <= 1e-12 * size + ulp * np.max(np.abs(ref))


@pytest.mark.parametrize("N,dtype", [(64, "f64"), (256, "f64"), (320, "f64"), (384, "f64"), (512, "f64"),
                                     (640, "f32"), (768, "f32"), (1024, "f32")])
def test_waves_of_known_power(N, dtype):
    waves = [(N // 2 - 1, 1, N // 4 + 1), (3, -(N // 2 - 2), 5), (0, 0, 7), (1, N // 8, -(N // 3))]
    npd, cd = (np.float32, np.complex64) if dtype == "f32" else (np.float64, np.complex128)
    f = np.zeros((N, N, N), npd)
    x = np.arange(N)
    for i, n in enumerate(waves):  # cos(2 pi n.r / N + i), array index [z][y][x]
        ex, ey, ez = (np.exp(2j * np.pi * ((c * x) % N) / N).astype(cd) for c in n)
        plane = (ey[:, None] * ex[None, :]) * cd(np.exp(1j * i))
        for z in range(N):
            f[z] += plane.real * ez[z].real - plane.imag * ez[z].imag
    with T.Lattice(N, 2 * np.pi, 1, dtype) as lat:  # a box of volume 1
        lat.set_state(f[None], f[None])
        k, P, c = lat.spectrum(0, 0)
    power = np.zeros(len(P))
    for n in waves:
        power[int(np.floor(np.sqrt(sum(v * v for v in n)) + 0.5))] += 0.5  # 1/4 at n and at -n
    # a wave's values are stored to a few ulp, so every mode is off by a few ulp of an
    # amplitude at most, and all together by as much of the total power
    ulp = 2.0 ** -52 if dtype == "f64" else 2.0 ** -23
    assert np.max(np.abs(P * c - power)) <= 32 * ulp


@pytest.mark.parametrize("N,dtype", [(256, "f64"), (320, "f64"), (384, "f64"), (512, "f64"), (640, "f32"),
                                     (768, "f32"), (1024, "f32")])
def test_drawn_modulus_is_measured(N, dtype):
    """A field of fixed modulus: every mode with 0 < |n| < N/2 has power A/(2 omega)."""
    kIR, m2, A = 0.5, 2.0, 1e-2
    with T.Lattice(N, kIR, 1, dtype) as lat:
        lat.set_potential(1.0, 0.0, (0.0, 0.0, 0.0))
        lat.init_fluctuations(7, A=A, meff2=(m2, 0, 0), phi0=(0.0, 0, 0), fixed_modulus=True)
        k, P, c = lat.spectrum(0, 0)
    g = np.arange(-10, 11)
    r2 = (g[:, None, None] ** 2 + g[None, :, None] ** 2 + g[None, None, :] ** 2).ravel()
    b = np.floor(np.sqrt(r2) + 0.5).astype(int)
    tol = 1e-12 if dtype == "f64" else 1e-5
    for s in range(1, 9):
        want = np.mean(A / (2.0 * np.sqrt(kIR ** 2 * r2[b == s] + m2)))
        assert abs(P[s] - want) <= tol * want
    assert np.all(P[N // 2 + 2:] <= tol ** 2 * P[1])
