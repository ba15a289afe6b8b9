"""Counts of valid anchors for flags that start anywhere, by the threshold on visible anchors (a fraction of
1 needs all of them), in the plain, batched and served forms."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 3, 8, 15])
@pytest.mark.parametrize("n", [1, 15, 16, 33, 400, 10000])
def test_threshold(shift, n):
    """Every valid anchor is seen from the ground truth, so a threshold of all of them is met exactly, and
    missed with one of them out of sight; the bytes beside the flags are set too."""
    torch = require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=100, n_hyps=1, levels=((240, 320),)), 81)
    seen = np.flatnonzero(f.point_valid)
    keep = np.concatenate([seen[:(n + 1) // 2], seen[:n // 2]])[:n]
    keep = np.resize(keep, n)
    arrs = B.device_arrays(f)
    flags = torch.ones(n + 64, dtype=torch.uint8, device="cuda")
    valid = flags[16 + shift:16 + shift + n]
    k = max(1, n - n // 3)
    valid[k:] = 0
    T = torch.as_tensor(np.ascontiguousarray(f.T_gt).reshape(1, 12), device="cuda")
    i = torch.as_tensor(keep, device="cuda")
    arrs.update(points=arrs["points"][:, i].contiguous(), point_weight=arrs["point_weight"][i].contiguous(), point_valid=valid,
                ref_feat=[arrs["ref_feat"][0][i].contiguous()], T_cw=T)
    fa = B.FrameArgs(f, arrs, is_device=True)
    opts = B.Options(iters=(0, 0, 0, 0), min_valid_frac=1.0, max_points=max(n, 64), max_hyps=1, max_frames=1)
    s, server = B.Solver(opts), B.Server(opts, 1 << 30, 1)
    for r in (s.solve(fa), s.solve_batch([fa])[0], server.wait(server.submit(fa))[0]):
        assert r.n_valid[0] == k and r.status[0] == B.HYP_OK
    arrs["points"][:, 0] = torch.as_tensor([0.0, 0.0, 1e6], device="cuda")       # behind the camera
    for r in (s.solve(fa), s.solve_batch([fa])[0], server.wait(server.submit(fa))[0]):
        assert r.n_valid[0] == k - 1 and r.status[0] == B.HYP_FEW_VALID
    s.close(), server.close()
