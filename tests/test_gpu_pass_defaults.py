"""Default launch shapes of the fused pass, alone and in a batch, against one
plain streaming shape: thin FP64 chunks with fewer rows than fit, FP32 chunks of
one wave, TMA tiles whose rows are cut in equal parts (with one, two and three
fields, 7 and 15 compute warps), the TMA shape of batch members.  On a static
background the fields are bitwise the same whatever the shape; the energy sums
differ by the rounding of their order.  And the scale factor's powers for whole
and fractional alpha against the oracle."""
import numpy as np
import pytest

import oracle as o
from paper_2607_24908_gb300 import tl as T
from paper_2607_24908_gb300.workloads import white_noise_state

pytestmark = pytest.mark.gpu

M2 = (0.0, 0.2, 0.1)
PLAIN = dict(kind="stream", z_chunk=16)


def lattice(N, nf, dtype, seed, alpha=1.0, expanding=False):
    npd = np.float32 if dtype == "f32" else np.float64
    phi, pi = white_noise_state(N, nf, seed=seed, phi0=(1.0, 0.0, 0.0)[:nf], sigma_phi=1e-2, sigma_pi=1e-2)
    lat = T.Lattice(N, 0.5, nf, dtype, expanding, alpha, 1.0, 1.0)
    lat.set_potential(1.0, 10.0, M2)
    lat.set_state(phi.astype(npd), pi.astype(npd), 1.0, 0.0, b_from_constraint=expanding)
    return lat, phi, pi


def run(N, nf, dtype, shape, seed=3, steps=4):
    lat, _, _ = lattice(N, nf, dtype, seed)
    with lat:
        if shape:
            lat.set_pass_config(**shape)
        lat.step(steps, 0.01, "verlet")
        return (*lat.get_all(), lat.energies().vector())


def same(got, ref, dtype):
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    tol = 1e-5 if dtype == "f32" else 1e-12
    assert np.max(np.abs(got[2] - ref[2])) <= tol * np.sum(np.abs(ref[2]))


@pytest.mark.parametrize("N,nf,dtype", [
    (8, 1, "f64"), (12, 1, "f64"), (20, 3, "f64"), (32, 1, "f64"), (60, 2, "f64"), (96, 1, "f64"),
    (8, 3, "f32"), (48, 2, "f32"), (76, 3, "f32"), (160, 2, "f32"), (188, 1, "f32"),
    (192, 3, "f32"), (200, 3, "f32"), (212, 1, "f32"), (260, 2, "f32"), (260, 3, "f32"), (396, 1, "f32")])
def test_default_shape_equals_plain_streaming(N, nf, dtype):
    same(run(N, nf, dtype, None), run(N, nf, dtype, PLAIN if N >= 16 else dict(kind="stream", z_chunk=N)), dtype)


@pytest.mark.parametrize("N,nf,zc,tile_x", [(8, 2, 3, 0), (12, 1, 5, 0), (20, 2, 20, 0), (36, 1, 16, 8), (68, 1, 17, 0),
                                            (68, 2, 33, 16), (100, 1, 3, 0), (100, 2, 50, 8), (132, 1, 48, 0), (20, 3, 4, 0),
                                            (76, 3, 34, 0)])
def test_shared_planes_equal_plain_streaming(N, nf, zc, tile_x):
    """FP64 with planes in shared memory (256 threads) against 512 threads, which
    read their neighbours from memory: tiles cut by both edges of the lattice, rows
    that straddle warps, chunks around the three planes of the ring and the 16 of
    a sum, the last one short."""
    got = run(N, nf, "f64", dict(kind="stream", z_chunk=zc, tile_x=tile_x))
    same(got, run(N, nf, "f64", dict(kind="stream", z_chunk=min(16, N), threads=512)), "f64")


@pytest.mark.parametrize("nf", [1, 2, 3])
@pytest.mark.parametrize("shape", [dict(kind="tma", warps=7, z_chunk=17), dict(kind="tma", warps=15, z_chunk=40)],
                         ids=["7-17", "15-40"])
def test_tma_tiles_inside_and_at_the_edge(nf, shape):
    """268 = 67 vectors a row: tiles of unequal width, the last one short, and
    tiles that touch no border of the lattice."""
    same(run(268, nf, "f32", shape), run(268, nf, "f32", PLAIN), "f32")


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("sizes", [(76, 80, 96), (80, 100, 192), (16, 36)], ids=str)
def test_batch_members_equal_plain_streaming(sizes, dtype):
    members = [(N, nf) for N in sizes for nf in (1, 2, 3)]
    lats = [lattice(N, nf, dtype, 7 + i)[0] for i, (N, nf) in enumerate(members)]
    with T.Batch(lats) as b:
        b.step(4, 0.01, "verlet")
    for i, (lat, (N, nf)) in enumerate(zip(lats, members)):
        with lat:
            same((*lat.get_all(), lat.energies().vector()), run(N, nf, dtype, PLAIN, 7 + i), dtype)


@pytest.mark.parametrize("alpha", [-1.0, 0.0, 0.5, 1.0, 2.0, 1.0 / 3.0])
def test_scale_powers_against_oracle(alpha):
    N, nf, steps, dt = 12, 2, 6, 0.01
    lat, phi0, pi0 = lattice(N, nf, "f64", 11, alpha, True)
    p = o.Params(N=N, nf=nf, kIR=0.5, expanding=True, alpha=alpha, lam=1.0, q=10.0, m2=M2)
    with lat:
        lat.step(steps, dt, "verlet")
        phi, pi = lat.get_all()
        E = lat.energies()
    b0 = np.sqrt(np.sum(o.energies(p, phi0, pi0, 1.0)) / 3.0)
    ophi, opi, oa, ob = o.run(p, phi0, pi0, 1.0, b0, dt, steps, o.VERLET)
    assert np.max(np.abs(phi - ophi)) / np.max(np.abs(ophi)) < 1e-12
    assert np.max(np.abs(pi - opi)) / np.max(np.abs(opi)) < 1e-12
    assert abs(E.a - oa) / oa < 1e-12 and abs(E.b - ob) / ob < 1e-12
