"""Levels of small frames run in one launch (one hypothesis or four per CTA, one or several anchor
tiles per cluster; batched: job tiles claimed for a whole level): every output bitwise that of the
batched form in lockstep (which a frame of two anchor tiles in the batch asks for), over storage types, channels, scales, confidence maps and the
sizes at which the layout changes (batches of 64 anchors, steps of 256, tiles of 1024)."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_cuda()


@pytest.fixture(scope="module")
def frames():
    made = {}

    def get(C, n_hyps=160):
        if C not in made:
            cfg = S.config_reduced_frame(crop_side=96, n_hyps=n_hyps, channels=C, levels=((120, 160), (60, 80)), f0=300.0)
            made[C] = S.with_query_confidence(S.make_frame(cfg, 31 + C), 7)
        return made[C]
    return get


def cut(frame, n, m, conf):
    """The frame's first n anchors (of a shuffled order, so that they spread over the crop) and m hypotheses."""
    keep = np.random.default_rng(5).permutation(frame.N)[:n]
    return frame.replace(points=np.ascontiguousarray(frame.points[:, keep]), point_valid=frame.point_valid[keep],
                         point_weight=(0.5 + np.arange(n, dtype=np.float32) % 7 / 7.0),
                         ref_feat=[np.ascontiguousarray(f[keep]) for f in frame.ref_feat], T_hyps=frame.T_hyps[:m],
                         qry_conf=frame.qry_conf if conf else None)


def check(torch, frame, dt, per_channel, damping=0):
    opts = B.Options(iters=(3, 2), max_points=max(frame.N, 1100), max_hyps=frame.M + 1, max_channels=frame.C, max_frames=2,
                     damping_mode=damping, keep_top_k=(0, max(1, frame.M // 2), 0, 0))
    fa = B.FrameArgs(frame, B.quantized_device_arrays(frame, dt, per_channel=per_channel), is_device=True, dtype=dt)
    # a second frame of 1100 anchors sends the batch through the lockstep schedule
    two = frame.replace(points=np.resize(frame.points[:, :1], (3, 1100)), point_valid=np.ones(1100, np.uint8),
                        point_weight=np.ones(1100, np.float32),
                        ref_feat=[np.resize(f[:1], (1100, frame.C)) for f in frame.ref_feat], T_hyps=frame.T_hyps[:1])
    fb = B.FrameArgs(two, B.quantized_device_arrays(two, dt, per_channel=per_channel), is_device=True, dtype=dt)
    s = B.Solver(opts)
    a = s.solve(fa)
    for b in (s.solve_batch([fa])[0], s.solve_batch([fa, fb])[0]):
        np.testing.assert_array_equal(a.T_cw, b.T_cw)
        np.testing.assert_array_equal(a.cost, b.cost)
        np.testing.assert_array_equal(a.n_valid, b.n_valid)
        np.testing.assert_array_equal(a.status, b.status)
        assert a.best == b.best
    # the evaluation of one level, with and without a handle
    T = np.ascontiguousarray(frame.T_hyps)
    ne = s.normal_eq(fa, 1, T)
    out = torch.zeros((frame.M, 29), dtype=torch.float64, device="cuda")
    assert B.normal_eq_noalloc(opts, fa, 1, torch.as_tensor(T, device="cuda"), out) == B.PILOT_OK
    torch.cuda.synchronize()
    np.testing.assert_array_equal(ne, out.cpu().numpy())
    s.close()
    return a


@pytest.mark.parametrize("n", [1, 63, 64, 65, 255, 256, 257, 500, 1023, 1024, 1025, 2049, 4097, 8192, 8193])
@pytest.mark.parametrize("m", [1, 19])
def test_anchor_counts(torch, frames, n, m):
    check(torch, cut(frames(32), n, m, False), B.F32, False)


@pytest.mark.parametrize("m", [2, 5, 76, 77, 152, 153, 160])
def test_hypothesis_counts(torch, frames, m):
    check(torch, cut(frames(32), 700, m, False), B.BF16, False)
    check(torch, cut(frames(32), 1500, m, True), B.F32, False, damping=1)


@pytest.mark.parametrize("C", [4, 8, 16, 32, 64])
@pytest.mark.parametrize("dt,per_channel", [(B.F32, False), (B.BF16, False), (B.BF16, True), (B.F16, False),
                                            (B.F16, True), (B.FP8E4M3, True)])
def test_storage_types(torch, frames, C, dt, per_channel):
    for conf in (False, True):
        r = check(torch, cut(frames(C), 1301, 9, conf), dt, per_channel)
        assert np.isfinite(r.cost).all()


def test_f32_scales_and_non_finite_maps(torch, frames):
    f = cut(frames(32), 600, 7, False)
    arrs = B.device_arrays(f)
    ones = torch.linspace(0.5, 1.5, 32, device="cuda")
    arrs.update(qry_scale=[ones, ones], ref_scale=[ones, ones])
    for poison in (False, True):
        if poison:
            arrs["qry_feat"][1][10:40, 20:60, 3] = float("nan")
            arrs["qry_feat"][0][50, :, 5] = float("inf")
        fa = B.FrameArgs(f, arrs, is_device=True)
        s = B.Solver(B.Options(iters=(3, 2), max_points=600, max_hyps=7, max_frames=1))
        a, b = s.solve(fa), s.solve_batch([fa])[0]
        np.testing.assert_array_equal(a.T_cw, b.T_cw)
        np.testing.assert_array_equal(a.cost, b.cost)
        np.testing.assert_array_equal(a.status, b.status)
        s.close()


@pytest.mark.parametrize("m,n", [(15, 8000), (16, 8000), (76, 2000), (77, 2000), (116, 7500), (117, 7500), (152, 1000)])
def test_lines_between_the_forms(torch, frames, m, n):
    """Around the hypotheses x tiles at which a level leaves one CTA per hypothesis, and one launch."""
    check(torch, cut(frames(32), n, m, False), B.F32, False)
