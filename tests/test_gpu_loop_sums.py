"""The grid-wide sums of the one-launch iteration loop (Cov, FP32) carry FP64's 53 bits, as those
of the other form (fused_tail 1) do.  S = I and a diagonal Omega whose squares have 24 bits
at three scales: a warp's sums are exact in its FP32 pair, the sum over all rows has 53 bits,
so that it is exact in FP64 and both forms have to return the same objective."""
import numpy as np
import pytest
from scipy.linalg import hadamard

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_objective_has_all_bits(lib, seed):
    import torch

    p = 1024
    X = torch.as_tensor(hadamard(p).astype(np.float32)).cuda()
    w = 1.0 + np.random.default_rng(seed).integers(0, 2048, p) / 2048.0
    w[:352] *= 2.0 ** 6
    w[704:] *= 2.0 ** -4
    om = lib.Csr(np.arange(p + 1), np.arange(p, dtype=np.int32), w)
    F = []
    for tail in (0, 1):
        with lib.Solver(X, 0.5, 0.125, precision=lib.PREC_FP32) as s:
            s.set_tuning(fused_tail=tail)
            s.set_omega(om)
            F.append(s.iterate(1).F)
    assert F[0] == F[1], (F, F[0] - F[1])
    # the parts that need no logarithm, exactly, and the logarithms of FP32
    exact = 0.5 * 1.125 * float(np.sum(w * w)) - float(np.sum(np.log(w.astype(np.float32)).astype(np.float64)))
    assert F[0] == pytest.approx(exact, rel=1e-9)
