"""The one-launch iteration loop of FP64 handles at its smallest sizes (224 rows on) against the
fused tail and the host-driven loop: the same iterates bit for bit."""
import numpy as np
import pytest

from workloads import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,lam1", [(224, 90, 0.2), (252, 92, 0.5), (257, 130, 0.12), (383, 200, 0.1)])
def test_small_fp64_loop(lib, p, n, lam1):
    import torch

    X = torch.as_tensor(small_problem(p, n, 4.0, seed=p).astype(np.float64)).cuda()
    out = []
    for tail, loop in ((0, 1), (1, 1), (0, 0)):
        with lib.Solver(X, lam1, 0.1, value_dtype=lib.F64, precision=lib.PREC_FP64, eps=1e-9, max_iter=20000,
                        device_loop=loop) as s:
            s.set_tuning(fused_tail=tail)
            out.append((s.solve().as_dict(), s.get_omega()))
    for st, om in out[1:]:
        assert (st["iterations"], st["ls_trials"], st["nnz"], st["status"]) == \
            tuple(out[0][0][k] for k in ("iterations", "ls_trials", "nnz", "status"))
        assert all(np.array_equal(getattr(om, f), getattr(out[0][1], f)) for f in ("row_ptr", "col", "val"))
        assert st["F"] == pytest.approx(out[0][0]["F"], rel=1e-11)
