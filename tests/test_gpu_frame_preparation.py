"""The calls around the solver at the sizes where their kernels change path: the quantiser's
channel counts (a thread's channels fixed or not) and store widths, the anchor draw's kept and
re-hashed keys and its further digits, and the crop's cell sizes that are no power of two."""
import ctypes as ct

import numpy as np
import pytest

from oracle import crop as OC
from oracle import sampler as OS
from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda
from precision_support import encode_bf16_rne, encode_e4m3_satfinite

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_cuda()


@pytest.mark.parametrize("dt", [B.BF16, B.F16, B.FP8E4M3])
@pytest.mark.parametrize("rows,C,per_channel,shift", [(1, 4, True, 0), (37, 12, True, 0), (1001, 64, True, 1),
                                                      (513, 1024, True, 0), (300, 2048, True, 1), (777, 20, False, 1),
                                                      (20000, 32, False, 0), (0, 8, True, 0)])
def test_quantiser_paths(torch, dt, rows, C, per_channel, shift):
    """Bit-exact against the format definitions; `shift` words off an 8-byte boundary for dst."""
    rng = np.random.default_rng(rows + C)
    x = (rng.standard_normal((rows, C)) * rng.uniform(0.01, 3.0, C)).astype(np.float32)
    if rows:
        x[:, 1] = 0.0                                     # a channel without a scale
        x[0, 0] = -0.0
    es = 1 if dt == B.FP8E4M3 else 2
    src = torch.zeros(rows * C + 4, device="cuda")       # an empty tensor has no address
    src[:rows * C] = torch.as_tensor(x.ravel(), device="cuda")
    dst = torch.zeros(rows * C * es + 16, dtype=torch.uint8, device="cuda")
    scale = torch.full((C,), 7.0, device="cuda")
    B.check(B.load().pilot_quantize_features(src.data_ptr(), rows, C, dt, int(per_channel),
                                             ct.c_void_p(dst.data_ptr() + 4 * shift), scale.data_ptr(),
                                             torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    want_s = np.ones(C, np.float32)
    if rows and (per_channel or dt == B.FP8E4M3):
        qmax = np.float32({B.FP8E4M3: 448.0, B.F16: 65504.0, B.BF16: 1.0}[dt])
        amax = np.abs(x).max(axis=0)
        want_s = np.where(amax > 0, (amax / qmax).astype(np.float32), np.float32(1.0))
    np.testing.assert_array_equal(scale.cpu().numpy(), want_s)
    y = x * (np.float32(1.0) / want_s)
    got = dst.cpu().numpy()
    body = got[4 * shift:4 * shift + rows * C * es]
    want = (encode_bf16_rne(y) if dt == B.BF16 else y.astype(np.float16).view(np.uint16) if dt == B.F16
            else encode_e4m3_satfinite(y))
    np.testing.assert_array_equal(body.view(want.dtype).reshape(rows, C), want)
    assert not got[:4 * shift].any() and not got[4 * shift + rows * C * es:].any()     # nothing beside it


@pytest.mark.parametrize("n,frac,k", [(65536, 0.9, 500), (65537, 0.5, 3000), (163840, 1.0, 1), (163841, 0.7, 2000),
                                      (3_000_000, 0.9, 5000), (4096, 1.0, 4095), (4096, 0.5, 4096), (31, 0.5, 8),
                                      (1, 0.0, 5), (5000, 0.0, 5)])
def test_anchor_draw_paths(torch, n, frac, k):
    rng = np.random.default_rng(n)
    valid = rng.random(n) < frac
    pts = rng.standard_normal((3, n)).astype(np.float32)
    v = torch.as_tensor(valid.astype(np.uint8), device="cuda")
    out = B.sample_anchors(v, torch.as_tensor(pts, device="cuda"), k, 90 + n)
    torch.cuda.synchronize()
    z = (np.uint64(90 + n) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    key = ((z ^ (z >> np.uint64(31))) >> np.uint64(32) << np.uint64(32)) | np.arange(n, dtype=np.uint64)
    j = np.nonzero(valid)[0]
    want = np.sort(j[np.argsort(key[j])][:k])
    if 0 < n <= 70000:                                    # the vectorised draw above is the oracle's
        np.testing.assert_array_equal(want, OS.sample_anchors(valid, k, 90 + n))
    c = int(out["count"].item())
    assert c == len(want)
    np.testing.assert_array_equal(out["idx"][:c].cpu().numpy(), want)
    np.testing.assert_array_equal(out["points"][:, :c].cpu().numpy(), pts[:, want])
    assert (out["idx"][c:] == -1).all() and not out["points"][:, c:].any()


@pytest.mark.parametrize("gsd,S_", [(0.3, 97), (0.7, 130), (1.0 / 3.0, 64)])
def test_crop_cell_sizes(torch, gsd, S_):
    g = S.make_global_map(side=1024, gsd=gsd, n_hills=128, n_boxes=256, seed=4)
    dm = B.MapArgs(torch.as_tensor(g.dsm, device="cuda"), torch.as_tensor(g.tdom, device="cuda"), g.x0, g.y0, g.gsd)
    om = OC.MapArgs(g.dsm, g.tdom, g.x0, g.y0, g.gsd)
    pr = S.crop_prior(g, 2, margin=0.35 * 1024 * gsd, altitude=(60.0, 80.0), pitch_deg=(60.0, 75.0))
    args = (pr["T_cw"], pr["fx"], pr["fy"], pr["cx"], pr["cy"], pr["img_w"], pr["img_h"], 0.0, 0.1, 3000, S_)
    o = OC.crop(om, OC.params(*args))
    d = B.crop_reference(dm, B.crop_params(*args))
    torch.cuda.synchronize()
    geo = d["geometry"].cpu().numpy()
    np.testing.assert_array_equal(geo[23:27].astype(int), o["idx"])
    assert bool(geo[27]) == o["ok"] and o["ok"]
    np.testing.assert_allclose(geo[:9], o["H"], rtol=1e-9, atol=1e-9)
    np.testing.assert_array_equal(d["valid"].cpu().numpy(), o["valid"])
    np.testing.assert_allclose(d["points"].cpu().numpy(), o["points"], atol=1e-4)
    np.testing.assert_allclose(d["rgb"].cpu().numpy(), o["rgb"], atol=1e-3)
