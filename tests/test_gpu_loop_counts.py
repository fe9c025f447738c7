"""hpc_stats.candidates, the entries that the screening emits: the one-launch loop counts as the chain of
kernels does, with up to half of the rows having neighbours (two rows with the diagonal alone
emit both entries of a pair, or none) and with more (each row its own)."""
import numpy as np
import pytest

from workloads import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,lam1,f64", [(600, 400, 0.15, False), (1217, 500, 0.15, False), (900, 400, 0.3, False),
                                          (450, 300, 0.15, True), (450, 300, 0.35, True)])
def test_candidates_at_every_iteration(lib, p, n, lam1, f64):
    import torch

    X = torch.as_tensor(small_problem(p, n, 4.0, seed=p).astype(np.float64 if f64 else np.float32)).cuda()
    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64) if f64 else dict(precision=lib.PREC_FP32)
    got = []
    for tail in (0, 1):
        with lib.Solver(X, lam1, 0.1, **opt) as s:
            s.set_tuning(fused_tail=tail)
            got.append([(d["candidates"], d["nnz"]) for d in (s.iterate(1).as_dict() for _ in range(16))])
    assert got[0] == got[1]
