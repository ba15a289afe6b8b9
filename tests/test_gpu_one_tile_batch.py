"""Batches of one-tile frames.  The flag-wait self-test takes every batch with enough gather work
per job, these included (a batched solve of most of them has no flag to wait for, the self-test
has); either schedule gives the plain solve's results."""
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


@pytest.mark.parametrize("cut", [0, 1])
def test_frames_of_one_tile_and_one_work_item(cut):
    """4096 anchors in one tile (the schedule without grid barriers) and one less in one of two
    frames (job tiles claimed for the level): bitwise the plain solve's."""
    require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=64, n_hyps=9), S.frame_seed(2, 991))
    g = f if not cut else f.replace(points=np.ascontiguousarray(f.points[:, 1:]), point_valid=f.point_valid[1:],
                                    point_weight=f.point_weight[1:],
                                    ref_feat=[np.ascontiguousarray(r[1:]) for r in f.ref_feat])
    fas = [device_frame(f), device_frame(g)]
    solver = B.Solver(B.Options(iters=(3, 2, 2), max_points=4096, max_hyps=18, max_frames=2))
    solver.set_schedule(fas, True, tile=4096)
    for fa, r in zip(fas, solver.solve_batch(fas)):
        solver.set_schedule([fa], False, tile=4096)
        a = solver.solve(fa)
        np.testing.assert_array_equal(a.T_cw, r.T_cw)
        np.testing.assert_array_equal(a.cost, r.cost)
        np.testing.assert_array_equal(a.status, r.status)
    solver.close()
