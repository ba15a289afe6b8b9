"""The reference crop at the sides where its CTA size changes: one warp per sub-partition, one CTA per
SM of growing size, the largest CTA, many CTAs per SM; against the FP64 oracle."""
import numpy as np
import pytest

from oracle import crop as OC
from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def maps():
    torch = require_cuda()
    g = S.make_global_map(side=1024, gsd=0.5, n_hills=128, n_boxes=256, seed=22)
    return (g, OC.MapArgs(g.dsm, g.tdom, g.x0, g.y0, g.gsd),
            B.MapArgs(torch.as_tensor(g.dsm, device="cuda"), torch.as_tensor(g.tdom, device="cuda"), g.x0, g.y0, g.gsd))


# warps per SM (152 SMs): 128^2 4, 140^2 5, 394^2 32, 395^2 33
@pytest.mark.parametrize("side", [1, 5, 64, 139, 140, 256, 394, 395, 600])
def test_crop_sides(maps, side):
    g, om, dm = maps
    pr = S.crop_prior(g, 3, margin=150.0, altitude=(80.0, 120.0), pitch_deg=(45.0, 70.0))
    args = (pr["T_cw"], pr["fx"], pr["fy"], pr["cx"], pr["cy"], pr["img_w"], pr["img_h"], 0.0, 0.25, 4000, side)
    o = OC.crop(om, OC.params(*args))
    n = side * side
    import torch
    out = dict(points=torch.full((3 * n + 64,), -7.0, device="cuda"), valid=torch.full((n + 64,), 9, device="cuda", dtype=torch.uint8),
               rgb=torch.full((3 * n + 64,), -7.0, device="cuda"), geometry=torch.empty(28, device="cuda", dtype=torch.float64))
    B.crop_reference(dm, B.crop_params(*args), out=out)
    torch.cuda.synchronize()
    assert o["ok"] and out["geometry"][27] == 1.0
    valid, pts, rgb = (out[k].cpu().numpy() for k in ("valid", "points", "rgb"))
    np.testing.assert_array_equal(valid[:n], o["valid"])
    p = pts[:3 * n].reshape(3, n)
    np.testing.assert_allclose(p[:2], o["points"][:2], atol=1e-4)      # FP32 roundings of the same doubles
    np.testing.assert_allclose(p[2], o["points"][2], atol=1e-5)
    np.testing.assert_allclose(rgb[:3 * n].reshape(n, 3), o["rgb"], atol=1e-3)
    assert (valid[n:] == 9).all() and (pts[3 * n:] == -7).all() and (rgb[3 * n:] == -7).all()      # nothing beside it
