"""The quantiser over channel counts that do not divide a CTA's values: several steps per thread,
threads left over, more channels than a CTA has values; bit-exact against the format definitions."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B

from gpu_support import require_cuda
from precision_support import encode_bf16_rne, encode_e4m3_satfinite

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [B.BF16, B.F16, B.FP8E4M3])
@pytest.mark.parametrize("rows,C", [(400001, 12), (200003, 20), (90001, 48), (5, 52), (3001, 1028), (1201, 4092), (1, 4096), (1200, 2048)])
def test_any_channel_count(dt, rows, C):
    torch = require_cuda()
    rng = np.random.default_rng(rows + C)
    x = (rng.standard_normal((rows, C)) * rng.uniform(0.01, 3.0, C)).astype(np.float32)
    got, scale = B.quantize_features(torch.as_tensor(x, device="cuda"), dt, per_channel=True)
    qmax = np.float32({B.FP8E4M3: 448.0, B.F16: 65504.0, B.BF16: 1.0}[dt])
    want_s = (np.abs(x).max(axis=0) / qmax).astype(np.float32)
    np.testing.assert_array_equal(scale.cpu().numpy(), want_s)
    y = x * (np.float32(1.0) / want_s)
    want = (encode_bf16_rne(y) if dt == B.BF16 else y.astype(np.float16).view(np.uint16) if dt == B.F16
            else encode_e4m3_satfinite(y))
    np.testing.assert_array_equal(got.view(torch.uint8).cpu().numpy().view(want.dtype).reshape(rows, C), want)
