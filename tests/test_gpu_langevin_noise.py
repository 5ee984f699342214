"""The Langevin step's FP32 noise itself: from a zero field with unit noise and a unit
step the new field is the noise.  Both components of every pair are accurate
relative to themselves, also next to an axis of the circle, where one vanishes."""
import numpy as np
import pytest

import oracle as o
from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


def test_fp32_noise_keeps_its_relative_accuracy_next_to_the_axes():
    N, seed = 64, 31
    zero = np.zeros((1, N, N, N), np.float32)
    with T.Lattice(N, 0.5, 1, "f32") as lat:
        lat.set_state(zero, zero)
        lat.langevin(1, 1.0, 0.0, 0.0, 1.0, seed)
        xi = lat.get(0, 0).astype(np.float64).reshape(-1)
    words = o.philox2x64(np.arange(N ** 3 // 2, dtype=np.uint64), o.LANGEVIN_STREAM, seed)
    u1, u2 = o._uniforms(words)
    quarter = np.rint(4.0 * u2)
    rest = 2.0 * np.pi * (u2 - quarter / 4.0)  # the difference is exact
    c, s, q = np.cos(rest), np.sin(rest), quarter.astype(int) % 4
    cos = np.choose(q, [c, -s, -c, s])
    sin = np.choose(q, [s, c, -s, -c])
    r = np.sqrt(-2.0 * np.log(u1))
    # FP32 roundings (2^-24 each, relative).  Modulus: u1 and the logarithm (1 ulp: 2) count
    # 1/|ln u1| <= 1/ln 2 for u1 <= 1/2, halved by the root, the root: 3.2.  Angle: its
    # constant, product and sum: 3; the polynomial's last two operations: 2.  Product: 1
    keep = (u1 <= 0.5) & (cos != 0.0) & (sin != 0.0)
    tol = 9.2 * 2.0 ** -24
    for got, ref in ((xi[0::2], r * cos), (xi[1::2], r * sin)):
        assert np.max(np.abs(got[keep] / ref[keep] - 1.0)) <= tol
    assert np.min(np.abs(np.minimum(np.abs(cos), np.abs(sin)))[keep]) < 1e-4  # some are next to an axis
