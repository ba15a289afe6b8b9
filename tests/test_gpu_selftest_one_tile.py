"""The flag-wait self-test takes every batch with enough gather work per job, frames of one anchor
tile included (a batched solve of those has no flag to wait for, the self-test has)."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


def test_flag_timeout_on_one_tile_frames():
    require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=64, n_hyps=3), S.frame_seed(2, 990))
    fas = [device_frame(f)]
    solver = B.Solver(B.Options(max_points=4096, max_hyps=4, max_frames=1))
    solver.set_schedule(fas, True, tile=4096)                # 4096 anchors: one tile, one work item per job
    before = solver.solve_batch(fas)[0]
    ms = solver.selftest_flag_timeout(fas, 100.0)
    assert 90.0 <= ms < 5000.0
    after = solver.solve_batch(fas)[0]
    np.testing.assert_array_equal(before.T_cw, after.T_cw)
    np.testing.assert_array_equal(before.cost, after.cost)
    solver.close()
