"""Lattices are independent: two host threads that step SU(2) lattices of different
sizes, whose tiles need different amounts of shared memory of one kernel, each
get bitwise what the lattice gives alone."""
import threading

import numpy as np
import pytest

from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


def steps(N, dtype, seed, calls, out, start=None):
    with T.SU2(N, dtype) as lat:
        lat.init_random(seed, 0.4)
        if start:
            start.wait()
        for _ in range(calls):
            lat.step(1, 0.02)
        out[N, dtype] = lat.get_state()


@pytest.mark.parametrize("pair", [((33, "f64"), (100, "f64")), ((33, "f64"), (128, "f64")), ((33, "f32"), (100, "f32")),
                                  ((50, "f32"), (128, "f32")), ((33, "f32"), (128, "f64"))], ids=str)
def test_two_threads_step_lattices_of_two_sizes(pair):
    calls = 200
    alone, both = {}, {}
    for i, (N, dtype) in enumerate(pair):
        steps(N, dtype, 5 + i, calls, alone)
    start = threading.Barrier(2, timeout=120)
    threads = [threading.Thread(target=steps, args=(N, dtype, 5 + i, calls, both, start))
               for i, (N, dtype) in enumerate(pair)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for key in pair:
        assert key in both, f"{key} failed"
        for got, ref in zip(both[key], alone[key]):
            assert np.array_equal(got, ref), key
