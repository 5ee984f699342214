"""Initial fields and spectra over lattice sizes at which the half-size complex
transform's index pairs fall differently (the smallest lattices, N/4 odd and
even, sizes with odd factors, rows shorter and longer than a warp), against the
FP64 oracle."""
import numpy as np
import pytest

import oracle as o
from paper_2607_24908_gb300 import tl as T
from paper_2607_24908_gb300.workloads import white_noise_state

pytestmark = pytest.mark.gpu


def shell_means(N, kIR, nbins):
    """k of every shell summed in extended precision (a sequential FP64 sum over a
    shell, as the oracle's, is itself off by 1.4e-14 at N = 44)."""
    n = np.fft.fftfreq(N, 1.0 / N)
    r = np.sqrt((n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2).astype(np.longdouble)).ravel()
    b = np.floor(r + np.longdouble(0.5)).astype(int)
    total = np.zeros(nbins, np.longdouble)
    np.add.at(total, b, r)
    return np.longdouble(kIR) * total / np.maximum(np.bincount(b, minlength=nbins), 1)


@pytest.mark.parametrize("N", [8, 12, 16, 20, 44, 100, 132])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_spectrum_matches_oracle(N, dtype):
    npd = np.float32 if dtype == "f32" else np.float64
    phi, pi = white_noise_state(N, 1, seed=N, phi0=(0.5,), sigma_phi=0.1, sigma_pi=0.2)
    phi, pi = phi.astype(npd), pi.astype(npd)
    p = o.Params(N=N, nf=1, kIR=0.3)
    with T.Lattice(N, p.kIR, 1, dtype) as lat:
        lat.set_state(phi, pi)
        for which, arr in ((0, phi), (1, pi)):
            k, P, c = lat.spectrum(0, which)
            ok, oP, oc = o.spectrum(p, arr[0].astype(np.float64))
            assert np.array_equal(c, oc) and c.sum() == N ** 3
            ek = shell_means(N, p.kIR, len(k))
            assert np.max(np.abs(k - ek)) <= 1e-14 * np.max(ek)
            # |F|^2 to FFT rounding of the largest mode (the mean): 1e-14 of its amplitude, twice
            # that relative to the shell's own, and 1e-12 of the shell's power
            top = np.sqrt(np.max(oP))
            assert np.all(np.abs(P - oP) <= 1e-12 * oP + 2e-14 * top * np.sqrt(oP) + (1e-14 * top) ** 2)


@pytest.mark.parametrize("N", [8, 12, 20, 44, 64])
@pytest.mark.parametrize("fixed", [False, True])
def test_initial_fields_match_oracle(N, fixed):
    p = o.Params(N=N, nf=2, kIR=0.2, expanding=True, alpha=1.0, lam=1.0, q=10.0)
    spec = o.InitSpec(A=1e-8, meff2=(3.0, 10.0, 0), phi0=(1.0, 0.0, 0), fluct_pi=True, fixed_modulus=fixed)
    ophi, opi, _, ob = o.init_fluctuations(p, 5, spec)
    with T.Lattice(N, p.kIR, 2, "f64", True, 1.0, 1.0, 1.0) as lat:
        lat.set_potential(p.lam, p.q, (0, 0, 0))
        lat.init_fluctuations(5, A=1e-8, meff2=(3.0, 10.0, 0), phi0=(1.0, 0, 0), fluct_pi=True, fixed_modulus=fixed)
        phi, pi = lat.get_all()
        b = lat.energies().b
    # the fluctuation to 1e-12 of its size, plus one rounding of phi0 + fluctuation
    for got, ref, mean in ((phi[0], ophi[0], 1.0), (phi[1], ophi[1], 0.0), (pi[0], opi[0], 0.0), (pi[1], opi[1], 0.0)):
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref - mean)) + 2.0 ** -52 * mean
    assert abs(b - ob) <= 1e-12 * ob
