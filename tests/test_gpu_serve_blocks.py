"""Served frames over the block layouts of a round's set-up and finish: sixteen blocks per frame, fewer
with many slots, several frames per block; hypothesis counts that leave warps over.  Bitwise the
plain solve."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


def same(a, b):
    for k in ("T_cw", "cost", "n_valid", "status"):
        np.testing.assert_array_equal(getattr(a, k), getattr(b, k))
    assert a.best == b.best


@pytest.mark.parametrize("slots", [1, 257, 1500])
def test_hypothesis_counts(slots):
    require_cuda()
    cfg = S.config_reduced_frame(crop_side=16, n_hyps=1210, levels=((60, 80), (30, 40)), f0=150.0)
    f = S.make_frame(cfg, 77)
    opts = B.Options(iters=(2, 2, 0), keep_top_k=(0, 60, 0, 0), max_points=1024, max_hyps=1210, max_frames=1)
    solver, server = B.Solver(opts), B.Server(opts, 1 << 30, slots)
    for m in (1, 9, 129, 1210):
        g = device_frame(f.replace(T_hyps=f.T_hyps[:m]))
        same(server.wait(server.submit(g))[0], solver.solve(g))
    solver.close(), server.close()


def test_more_frames_than_blocks():
    """Frames that queue up behind a long round: more than 1024 run at once."""
    require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=8, n_hyps=1, levels=((60, 80),), f0=150.0), 78)
    g = device_frame(f)
    opts = B.Options(iters=(1500, 0, 0, 0), max_points=64, max_hyps=1500, max_frames=1)
    solver, server = B.Solver(opts), B.Server(opts, 1 << 30, 1500)
    want = solver.solve(g)
    results = [server.wait(t)[0] for t in [server.submit(g) for _ in range(2600)]]
    assert server.stats()["peak_active"] > 1024
    for r in results:
        same(r, want)
    solver.close(), server.close()
