"""Default launch shapes at sizes between the measured round ones: no slower than
the fixed shape (warps, planes) that the size's neighbourhood had before."""
import pytest

from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


def pass_ms(lat, steps):
    import torch

    lat.step(2, 1e-3)
    best = 1e9
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        lat.step(steps, 1e-3)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / (steps + 1))
    return best


@pytest.mark.parametrize("N,nf,warps,planes", [(340, 2, 7, 56), (340, 3, 7, 56), (372, 1, 15, 93), (420, 2, 15, 80),
                                               (652, 2, 15, 104), (772, 2, 15, 104)])
def test_default_is_not_slower_than_the_fixed_shape(N, nf, warps, planes):
    pytest.importorskip("torch")
    with T.Lattice(N, 0.1, nf, "f32") as lat:
        lat.set_potential(1.0, 10.0, (0.0, 0.2, 0.1))
        lat.init_fluctuations(1, A=0.0)  # uniform fields
        default = lat.pass_config()
        steps = 10
        ratio = 1e9
        for _ in range(3):  # up to 13% before; a few tries against a disturbed timing
            lat.set_pass_config(**default)
            mine = pass_ms(lat, steps)
            lat.set_pass_config("tma", warps=warps, z_chunk=planes)
            ratio = min(ratio, mine / pass_ms(lat, steps))
            if ratio <= 1.03:
                break
        assert ratio <= 1.03, (default, ratio)
