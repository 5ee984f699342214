"""The first initial fields of a size only enqueue work, as the later ones do: with
half a second of passes queued on the same stream the call returns at once.  Run in
a process of its own that loads every kernel up front (loading one on its
first launch waits for the device by itself)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
import time
from paper_2607_24908_gb300 import tl as T

def ready(N, nf=1, dtype="f32"):
    lat = T.Lattice(N, 0.5, nf, dtype)
    lat.set_potential(1.0, 10.0, (0.0, 0.2, 0.0))
    return lat

busy, warm, first = ready(256, 2, "f64"), ready(64), ready(128)
busy.init_fluctuations(1)
warm.init_fluctuations(2)
warm.energies()
busy.step(1, 1e-3)
busy.energies()
busy.step(400, 1e-3)        # about 1.2 ms a pass
t0 = time.perf_counter()
first.init_fluctuations(3)  # the first of its size
t1 = time.perf_counter()
busy.energies()             # waits for the passes
t2 = time.perf_counter()
first.energies()
print(t1 - t0, t2 - t1)
"""


def test_first_init_of_a_size_does_not_wait_for_its_stream():
    env = dict(os.environ, CUDA_MODULE_LOADING="EAGER", TL_STEP_GRAPHS="0", PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", MAIN], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    call, rest = (float(v) for v in out.stdout.split()[-2:])
    assert rest > 0.15, "the passes were done before the call could wait for them"
    assert call < 0.25 * (call + rest), (call, rest)
