"""Steps that run eight to a CUDA graph (handles and batches that keep stepping): no effect on a capture of
another stream while the graph is built."""
import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm
import synthetic

pytestmark = pytest.mark.gpu


def simulation(precision, nx, ny, stream=None):
    s = lbm.Simulation(nx, ny, lbm.default_params(precision=precision), stream=stream)
    s.init(*synthetic.spinodal(nx, ny, 1.0, 0.01, 0.9, seed=2))
    return s


def single_steps(precision, nx, ny, n):
    with simulation(precision, nx, ny) as s:
        s.timing(True)  # direct launches, no graph
        s.step(n)
        return s.get_f()


@pytest.mark.parametrize("mode", ["global", "thread_local"])
def test_graph_is_built_during_the_capture_of_another_stream(mode):
    import torch
    with simulation(lbm.LBM_MIXED, 64, 32, torch.cuda.Stream().cuda_stream) as s:
        s.step(33)
        s.synchronize()
        x, graph = torch.zeros(64, device="cuda"), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode=mode):
            y = x + 1
            s.step(8)
            z = y * 2
        graph.replay()
        torch.cuda.synchronize()
        assert float(z.sum()) == 128.0
        assert np.array_equal(s.get_f(), single_steps(lbm.LBM_MIXED, 64, 32, 41))
