"""Batches in handles for more frames than a launch has blocks side by side, and frames with more
hypotheses than its ranking takes in one turn: bitwise the plain solve of each frame."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def frame():
    require_cuda()
    return S.make_frame(S.config_reduced_frame(crop_side=8, n_hyps=1500, levels=((60, 80), (30, 40)), f0=150.0), 79)


@pytest.mark.parametrize("n,max_frames,counts", [(3, 65536, (9, 1500, 300)), (1030, 1030, (3, 9, 5)), (2100, 4096, (2, 1, 4))])
def test_frames_and_blocks(frame, n, max_frames, counts):
    fas = [device_frame(frame.replace(T_hyps=frame.T_hyps[:m])) for m in counts]
    opts = B.Options(iters=(2, 2, 0, 0), keep_top_k=(0, 2, 0, 0), max_points=512, max_hyps=8192, max_frames=max_frames)
    s = B.Solver(opts)
    want = [s.solve(fa) for fa in fas]
    got = s.solve_batch([fas[i % len(fas)] for i in range(n)])
    for i, r in enumerate(got):
        w = want[i % len(fas)]
        for k in ("T_cw", "cost", "n_valid", "status"):
            np.testing.assert_array_equal(getattr(r, k), getattr(w, k), err_msg=f"frame {i} {k}")
        assert r.best == w.best
    s.close()
