"""Plain solves of one anchor tile around the hypothesis count at which a level leaves the single launch
(304 CTAs of four): bitwise the batched form."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1216, 1217, 1300])
def test_one_tile_waves(m):
    require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=20, n_hyps=1300, levels=((60, 80), (30, 40)), f0=150.0), 82)
    fa = device_frame(f.replace(T_hyps=f.T_hyps[:m]))
    s = B.Solver(B.Options(iters=(3, 2, 0, 0), keep_top_k=(0, 1250, 0, 0), max_points=1024, max_hyps=m, max_frames=1))
    a, b = s.solve(fa), s.solve_batch([fa])[0]
    for k in ("T_cw", "cost", "n_valid", "status"):
        np.testing.assert_array_equal(getattr(a, k), getattr(b, k))
    assert a.best == b.best
    T = np.ascontiguousarray(f.T_hyps[:m])
    want = np.concatenate([s.normal_eq(device_frame(f.replace(T_hyps=T[i:i + 600])), 1, T[i:i + 600]) for i in range(0, m, 600)])
    np.testing.assert_array_equal(s.normal_eq(fa, 1, T), want)
    s.close()
