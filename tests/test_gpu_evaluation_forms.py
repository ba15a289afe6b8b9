"""One evaluation in its three forms (a pose per CTA, a hypothesis tile per CTA in clusters, a build pass
and an epilogue), by the number of poses: every pose's normal equations are bitwise the same."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,counts", [(90, (1, 15, 16, 76, 77, 116, 117)),     # 8 tiles
                                         (50, (1, 40, 41, 200, 201, 308, 309)),   # 3 tiles
                                         (30, (1, 152, 153, 400))])               # 1 tile
def test_forms_agree(side, counts):
    torch = require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=side, n_hyps=400), S.frame_seed(2, 995))
    s = B.Solver(B.Options(max_points=f.N, max_hyps=400, max_frames=1))
    want = None
    for m in sorted(counts, reverse=True):
        fa = device_frame(f.replace(T_hyps=f.T_hyps[:m]))
        got = s.normal_eq(fa, 0, f.T_hyps[:m])
        want = got if want is None else want
        np.testing.assert_array_equal(got, want[:m])
        if m <= 256:
            out = torch.zeros((m, 29), dtype=torch.float64, device="cuda")
            B.check(B.normal_eq_noalloc(B.Options(), fa, 0, fa.arrays["T_cw"], out))
            np.testing.assert_array_equal(out.cpu().numpy(), want[:m])
    s.close()
