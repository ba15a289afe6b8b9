"""Larger frames whose damped solves fail at first and succeed once lambda has grown: a hypothesis
tile without a candidate finds one in its step, and the launch's other CTAs of that tile, which may
start later, must not see it.  Bitwise the batched form, whose steps are published between
iterations."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_cuda()


@pytest.mark.parametrize("m", [1, 4, 5, 64])
@pytest.mark.parametrize("side", [104, 200])
def test_tiles_without_a_candidate(torch, side, m):
    """Every anchor is one point: the normal equations have rank 2, and the FP32 sums' rounding
    leaves a pivot below zero until lambda exceeds it."""
    f = S.make_frame(S.config_reduced_frame(crop_side=side, n_hyps=m), S.frame_seed(2, 980))
    f = f.replace(use_gravity=False, use_range=False)
    j = int(np.flatnonzero(f.point_valid)[f.point_valid.sum() // 2])
    arrs = B.device_arrays(f)
    arrs.update(points=arrs["points"][:, [j]].expand(3, f.N).contiguous(), point_valid=torch.ones_like(arrs["point_valid"]))
    arrs.update({k: arrs[k][:1] for k in ("qry_feat", "ref_feat")})
    fa = B.FrameArgs(f, arrs, is_device=True)
    start = arrs["T_cw"].cpu().numpy()
    res = {}
    for k in (3, 12, 25):
        s = B.Solver(B.Options(iters=(k,), lambda0=1e-12, min_valid_frac=0.0, max_points=f.N, max_hyps=m, max_frames=1))
        a = s.solve(fa)
        for b in (s.solve_batch([fa])[0], s.solve(fa)):
            np.testing.assert_array_equal(a.T_cw, b.T_cw)
            np.testing.assert_array_equal(a.cost, b.cost)
            np.testing.assert_array_equal(a.status, b.status)
        s.close()
        res[k] = a
    # whole tiles of hypotheses fail at first, and a later solve of theirs succeeds
    stuck = (res[3].status == B.HYP_NOT_PD) & (res[3].T_cw == start).all(axis=1)
    moved = (res[25].T_cw != start).any(axis=1)
    tiles = [range(i, min(i + 4, m)) for i in range(0, m, 4)]
    assert any(stuck[t].all() and moved[t].any() for t in tiles)
