"""Steps that run eight to a CUDA graph (handles and batches that keep stepping): the same bits however the
steps are split over calls, whatever drops the graph in between, and no effect on a capture of another
stream while the graph is built."""
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


@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_MIXED])
@pytest.mark.parametrize("calls", [[40, 24], [33, 8, 7, 16], [1] * 40 + [24], [300]])
def test_same_bits_however_split(precision, calls):
    with simulation(precision, 64, 32) as s:
        for n in calls:
            s.step(n)
        assert s.diagnostics()["steps"] == sum(calls)
        assert np.array_equal(s.get_f(), single_steps(precision, 64, 32, sum(calls)))


@pytest.mark.parametrize("change", ["geometry", "pass kinds", "fault injection off", "autotune", "diagnostics", "state"])
def test_changes_between_graphs(change):
    with simulation(lbm.LBM_MIXED, 128, 64) as s:
        s.step(40)
        s.step(16)
        if change == "geometry":
            g = list(s.geometry())
            s.set_geometry((max(4, g[0] // 2), g[1], g[2], max(4, g[3] // 2)))
        elif change == "pass kinds":
            s.set_pass_kinds((lbm.LBM_COL_DIRECT, lbm.LBM_COL_DIRECT, 1))
        elif change == "fault injection off":
            s.fault_inject(lbm.LBM_FAULT_NONE)
        elif change == "autotune":
            s.autotune()
        elif change == "diagnostics":
            s.diagnostics_begin()
        else:
            s.set_state(s.get_state())
        s.step(24)
        if change == "diagnostics":
            assert np.isfinite(s.diagnostics_end()["mass"])
        s.step(9)
        assert np.array_equal(s.get_f(), single_steps(lbm.LBM_MIXED, 128, 64, 89))


def test_batch_of_three_sizes():
    sizes = [(64, 64), (128, 32), (32, 64), (64, 64)]
    params = lbm.default_params(precision=lbm.LBM_MIXED)

    def run(calls):
        with lbm.Batch(sizes, params) as b:
            for k, (nx, ny) in enumerate(sizes):
                b.init(k, *synthetic.spinodal(nx, ny, 1.0, 0.01, 0.9, seed=k))
            for n in calls:
                b.step(n)
            return [b.get_f(k) for k in range(len(sizes))]

    one_by_one = run([7] * 42 + [6])
    for calls in ([40, 260], [300]):
        assert all(np.array_equal(a, b) for a, b in zip(one_by_one, run(calls)))


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
