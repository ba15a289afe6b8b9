"""Top-K of a plain solve at the hypothesis counts where a hypothesis' share of the ranking changes: the K
lowest objectives survive, ties by the lower index."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 255, 8192, 8193, 32768, 32769])
def test_survivors(m):
    require_cuda()
    f = S.make_frame(S.config_reduced_frame(crop_side=10, n_hyps=50, levels=((60, 80), (30, 40)), f0=150.0), 80)
    f = f.replace(T_hyps=np.resize(f.T_hyps, (m, 12)))          # every objective many times
    k = max(1, m // 7)
    s = B.Solver(B.Options(iters=(0, 0, 0, 0), keep_top_k=(0, k, 0, 0), min_valid_frac=0.0, max_points=512, max_hyps=m, max_frames=1))
    fa = device_frame(f)
    cost = s.normal_eq(fa, 1, f.T_hyps)[:, 27]
    r = s.solve(fa)
    keep = np.zeros(m, bool)
    keep[np.lexsort((np.arange(m), cost))[:k]] = True
    np.testing.assert_array_equal(r.status != B.HYP_PRUNED, keep)
    s.close()
