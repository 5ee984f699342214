"""Initial fields of a size whose table of roots exists can be captured into a CUDA
graph; the replay gives bitwise the fields of the direct call."""
import numpy as np
import pytest

from paper_2607_24908_gb300 import tl as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["global", "relaxed"])
def test_initial_fields_in_a_captured_stream(mode):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    with T.Lattice(64, 0.5, 1, "f32", True, 1.0, 1.0, 1.0, stream=stream.cuda_stream) as lat:
        lat.set_potential(1.0, 0.0)
        lat.init_fluctuations(7, 1e-3)
        ref = lat.get(0, 0)
        lat.init_fluctuations(8, 1e-3)
        assert not np.array_equal(lat.get(0, 0), ref)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode=mode):
            lat.init_fluctuations(7, 1e-3)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(lat.get(0, 0), ref)
        del graph
