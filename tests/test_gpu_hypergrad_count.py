"""hpc_hypergrad reports the CG iterations that it ran: with S_ii = 1 and Omega = I the Hessian on the
support is a multiple of the identity, so one iteration reaches the solution."""
import numpy as np
import pytest
from scipy.linalg import hadamard

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f64", [False, True])
def test_one_iteration(lib, f64):
    import torch

    p, n = 64, 128
    dtype = np.float64 if f64 else np.float32
    X = torch.as_tensor(hadamard(n)[:, :p].astype(dtype)).cuda()
    Xval = torch.as_tensor(np.random.default_rng(3).standard_normal((50, p)).astype(dtype)).cuda()
    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64) if f64 else dict(precision=lib.PREC_FP32)
    with lib.Solver(X, 0.2, 0.1, **opt) as s:
        d1, d2, info = s.hypergrad(Xval)
    assert info["converged"] == 1 and info["cg_iterations"] == 1, info
    assert d1 == 0.0
    b = (Xval.double().cpu().numpy() ** 2).mean(axis=0) - 1.0
    assert d2 == pytest.approx(-b.sum() / 2.1, rel=1e-5)
