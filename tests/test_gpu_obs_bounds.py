"""The Obs pass over the block pairs that its bounds keep: at every iterate the candidates and
the next iterate of a handle that has kept bounds since its load are those of a handle that
loads the data anew, sets the iterate and so takes every pair, bit for bit."""
import numpy as np
import pytest

from workloads import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,lam1,prec", [
    (100, 40, 0.2, "PREC_FP32"),        # one block: the diagonal pair alone
    (300, 100, 0.35, "PREC_FP32"),      # three ragged blocks, padded K steps
    (1200, 65, 0.5, "PREC_FP32"),       # ten blocks: a full band of the pair list and a part of one
    (1100, 130, 0.3, "PREC_TF32"),      # three K stages of BF16, five of TF32
    (1500, 100, 0.15, "PREC_FP32"),     # dense support
])
def test_kept_bounds_change_nothing(lib, p, n, lam1, prec):
    import torch

    X = torch.as_tensor(small_problem(p, n, 3.0, seed=p).astype(np.float32)).cuda()
    opt = dict(variant=lib.OBS, precision=getattr(lib, prec))
    with lib.Solver(X, lam1, 0.1, **opt) as a, lib.Solver(X, lam1, 0.1, **opt) as b:
        for step in range(14):
            if step == 9:       # another lambda1: pairs that were left out come back
                a.set_lambda(0.6 * lam1, 0.1)
                b.set_lambda(0.6 * lam1, 0.1)
            at = a.get_omega()
            b.load_x(X)
            b.set_omega(at)
            a.iterate(1)
            b.iterate(1)
            for x, y in zip(a.candidates(), b.candidates()):
                assert np.array_equal(x, y), step
            oa, ob = a.get_omega(), b.get_omega()
            assert np.array_equal(oa.row_ptr, ob.row_ptr) and np.array_equal(oa.col, ob.col), step
            assert np.array_equal(oa.val, ob.val), step
