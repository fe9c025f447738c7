"""The plain FP32 Gram at the edges of its tiles, K-slabs and dispatch, rows of X and S on and off
16-byte boundaries, against FP64 under the bound of an n-term FMA chain; S is bitwise symmetric."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,pad,xdt", [
    (1, 1, 0, "f32"), (64, 16, 0, "f32"), (63, 17, 0, "f32"), (65, 15, 3, "bf16"), (128, 33, 4, "bf16"),
    (129, 40, 0, "f64"), (260, 31, 1, "f32"),        # rows of S off 16 bytes
    (1620, 20, 0, "f32"), (1541, 20, 0, "f32"),      # 64 x 64 tiles, both loaders
    (1924, 20, 0, "bf16"), (1925, 20, 0, "f32"),     # 128 x 128 tiles, fewer than SMs
    (2200, 20, 0, "f32"),                            # a few more than SMs: 64 x 64 again
    (2501, 20, 0, "f64"), (2500, 20, 0, "f32"),
])
def test_plain_fp32_gram(lib, p, n, pad, xdt):
    import torch

    dt = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}[xdt]
    X = torch.randn((n, p), generator=torch.Generator().manual_seed(p + n), dtype=torch.float64).to(dt).cuda()
    buf = torch.full((p, p + pad), float("nan"), device="cuda")
    lib.gram(X, buf, precision=lib.PREC_FP32)
    S = buf[:, :p]
    Xd = X.float().double()
    bound = (n + 2) * 2.0 ** -24 * (Xd.abs().t() @ Xd.abs()) / n
    assert bool(((S.double() - Xd.t() @ Xd / n).abs() <= bound).all())
    assert torch.equal(S, S.t())
    assert bool(buf[:, p:].isnan().all())
