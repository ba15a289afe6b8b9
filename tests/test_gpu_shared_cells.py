"""The build pass reads a cell of the query map once for two hypotheses of an anchor that land in it:
whether they do, partly do (hypotheses that agree on some anchors, invisible ones) or don't, every
pose's sums are bitwise those of the pose evaluated alone, over the storage types, channel counts and
lane layouts."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_cuda()


def poses(frame):
    """Seventeen: agreeing, nearly agreeing, pixels apart, and out of view, in pairs of every kind."""
    base = np.array(frame.T_hyps[0], np.float64).reshape(3, 4)

    def shifted(d):
        T = base.copy()
        T[:, 3] += d
        return T.reshape(12)
    same, near = shifted([0, 0, 0]), shifted([3e-4, -2e-4, 1e-4])
    part, far = shifted([0.08, -0.05, 0.02]), shifted([6.0, 4.0, -2.0])
    gone, behind = shifted([1e5, 0, 0]), shifted([0, 0, -1e5])
    return np.array([same, same, same, same, near, same, part, near, far, same, gone, same, same, behind, gone, behind,
                     far])


def evaluate(torch, opts, fa, T):
    assert fa.M == len(T)
    out = torch.zeros((len(T), 29), dtype=torch.float64, device="cuda")
    assert B.normal_eq_noalloc(opts, fa, 0, torch.as_tensor(np.ascontiguousarray(T), device="cuda"), out) == B.PILOT_OK
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("C", [4, 8, 16, 32, 64])
@pytest.mark.parametrize("dt,per_channel", [(B.F32, False), (B.BF16, False), (B.F16, True), (B.FP8E4M3, True)])
@pytest.mark.parametrize("n,conf", [(8193, False), (9001, True)])
def test_sums_do_not_depend_on_the_other_hypotheses(torch, C, dt, per_channel, n, conf):
    cfg = S.config_reduced_frame(crop_side=96, n_hyps=17, channels=C, levels=((120, 160),), f0=300.0)
    frame = S.make_frame(cfg, 11)
    frame = S.with_query_confidence(frame, 7) if conf else frame
    keep = np.random.default_rng(3).permutation(frame.N)[:n]
    T = poses(frame)
    frame = frame.replace(points=np.ascontiguousarray(frame.points[:, keep]), point_valid=frame.point_valid[keep],
                          point_weight=frame.point_weight[keep], T_hyps=T,
                          ref_feat=[np.ascontiguousarray(f[keep]) for f in frame.ref_feat])
    arrays = B.quantized_device_arrays(frame, dt, per_channel=per_channel)
    opts = B.Options(iters=(1,), max_points=frame.N, max_hyps=17, max_channels=C, max_frames=1)
    together = evaluate(torch, opts, B.FrameArgs(frame, arrays, is_device=True, dtype=dt), T)
    assert np.isfinite(together).all() and (together[0] != 0).any()
    for order in (np.arange(17)[::-1], np.random.default_rng(1).permutation(17)):
        np.testing.assert_array_equal(evaluate(torch, opts, B.FrameArgs(frame, arrays, is_device=True, dtype=dt),
                                               T[order]), together[order])
    for m in (0, 4, 6, 8, 10, 13):
        one = B.FrameArgs(frame, dict(arrays, T_cw=arrays["T_cw"][m:m + 1]), is_device=True, dtype=dt)
        np.testing.assert_array_equal(evaluate(torch, opts, one, T[m:m + 1])[0], together[m])
