"""Column tiles of the float64 lines stay within what their reductions have room for (csrc/fft_line.cuh): 16
lines of a tile, 8 warps."""
import pytest

import paper_1403_3746_gb300 as lbm


@pytest.mark.parametrize("log2ny", range(1, 13))
def test_float64_column_tiles_fit_the_reductions(log2ny):
    for log2nx in range(1, 13):
        plan = lbm.launch_plan(1 << log2nx, 1 << log2ny, lbm.LBM_FP64)
        assert plan["col_width"] // 2 <= 16
        assert plan["col_threads"] <= 256 and plan["pass_thread_cap"] <= 256
