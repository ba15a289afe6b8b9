"""The anchor draw of small crops, which one CTA makes: around its largest size, around whole steps, with
all, none or one of the pixels taken; against the oracle's draw."""
import numpy as np
import pytest

from oracle import sampler as OS
from paper_2606_31098_gb300 import binding as B

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 1000, 1024, 1025, 4095, 4096, 4097])
@pytest.mark.parametrize("frac,select", [(1.0, "one less"), (0.6, "half"), (0.6, "all"), (0.6, "more"), (0.0, "half"), (0.9, 1), (0.9, 0)])
def test_small_draws(n, frac, select):
    torch = require_cuda()
    valid = np.random.default_rng(n).random(n) < frac
    count = int(valid.sum())
    k = {"one less": max(count - 1, 0), "half": n // 2, "all": count, "more": n + 7}.get(select, select)
    want = OS.sample_anchors(valid, k, 123 + n)
    pts = np.arange(3 * n, dtype=np.float32).reshape(3, n)
    out = dict(idx=torch.full((k + 4,), -1, dtype=torch.int32, device="cuda"),
               points=torch.zeros((3, max(k, 1)), device="cuda"), count=torch.full((1,), 9, dtype=torch.int32, device="cuda"))
    B.sample_anchors(torch.as_tensor(valid.astype(np.uint8), device="cuda"), torch.as_tensor(pts, device="cuda"), k, 123 + n, out=out)
    c = int(out["count"].item())
    assert c == len(want)
    np.testing.assert_array_equal(out["idx"][:c].cpu().numpy(), want)
    assert (out["idx"][c:] == -1).all()
    np.testing.assert_array_equal(out["points"][:, :c].cpu().numpy(), pts[:, want])
    assert not out["points"][:, c:].any()
