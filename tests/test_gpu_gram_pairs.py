"""Tensor-core Gram on CTA pairs (256 x 256 tiles; FP32 X): the edges of its tiles, of a
pair's halves (128 rows), of the K slabs and of the chunks of K, in both FP32 modes.

Bounds per entry as for the other tensor-core Gram tests, D_ij = sqrt(S_ii S_jj) and
u = 2^-24: BF16X3 (2^-15 + 2 n u) D, TF32 (2^-10 + 2 n u) D.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("mode,rel", [("PREC_BF16X3", 2.0 ** -15), ("PREC_TF32", 2.0 ** -10)])
@pytest.mark.parametrize("n,p", [(1, 129), (63, 255), (64, 256), (65, 257), (129, 384), (128, 385), (2113, 513)])
def test_tile_edges(lib, mode, rel, n, p):
    import torch

    rng = np.random.default_rng(7 * n + p)
    X = rng.standard_normal((n, p)).astype(np.float32)
    S = torch.full((p, p + 3), float("nan"), dtype=torch.float32, device="cuda")
    lib.gram(torch.as_tensor(X).cuda(), S, precision=getattr(lib, mode))
    torch.cuda.synchronize()
    got = S[:, :p].double().cpu().numpy()
    ref = oracle.gram(X.astype(np.float64))
    D = np.sqrt(np.outer(np.diag(ref), np.diag(ref)))
    assert np.all(np.abs(got - ref) <= (rel + 2 * n * U) * D)
    assert np.array_equal(got, got.T)
    assert torch.isnan(S[:, p:]).all()
