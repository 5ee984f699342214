"""tl_autotune chooses among shapes that include the one the lattice has: it never
leaves a lattice slower than it found it."""
import pytest

from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nf", [(212, 2), (224, 3)])
def test_autotune_does_not_slow_the_default_down(N, nf, monkeypatch):
    torch = pytest.importorskip("torch")
    monkeypatch.delenv("TL_TUNE_FILE", raising=False)

    def ms(lat, steps=20):
        lat.step(2, 1e-3)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            lat.step(steps, 1e-3)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    with T.Lattice(N, 0.1, nf, "f32") as lat:
        lat.set_potential(1.0, 10.0, (0.0, 0.2, 0.1))
        lat.init_fluctuations(1, A=0.0)
        before = ms(lat)
        lat.autotune()
        assert ms(lat) <= 1.08 * before  # 17% and 30% slower when the default was no candidate
