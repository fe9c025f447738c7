"""Forms of the one-launch loop's screening (Cov) against the other form of the iteration (fused_tail 1), at
every iterate: rows of more than 32 terms, the task list overflowing into the pass over all blocks
that the bounds keep, several pages of a row's bucket."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,lam1,k,f64", [
    (1000, 300, 0.1, 8, False),       # 60 to 90 entries a row
    (4096, 600, 0.1, 5, False),       # all 131 072 (row, block) tasks: the list holds 98 304
    (500, 200, 0.1, 8, True),
    (900, 2000, 0.02, 6, False),      # up to 400 candidates a row in some iterations
])
def test_every_iterate(lib, p, n, lam1, k, f64):
    import torch

    x = np.random.default_rng(p).standard_normal((n, p))
    x[:, 1:] += 0.4 * x[:, :-1]
    X = torch.as_tensor(x.astype(np.float64 if f64 else np.float32)).cuda()
    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64) if f64 else dict(precision=lib.PREC_FP32)
    out = []
    for tail in (0, 1):
        with lib.Solver(X, lam1, 0.1, **opt) as s:
            s.set_tuning(fused_tail=tail)
            runs = []
            for t in range(1, k + 1):
                s.load_x(X)
                st = s.iterate(t).as_dict()
                runs.append(([st[f] for f in ("iterations", "ls_trials", "nnz", "candidates")], st["F"], s.get_omega(),
                             s.candidates()))
            out.append(runs)
    for a, b in zip(*out):
        assert a[0] == b[0] and a[1] == pytest.approx(b[1], rel=1e-11)
        assert all(np.array_equal(getattr(a[2], f), getattr(b[2], f)) for f in ("row_ptr", "col", "val"))
        assert all(np.array_equal(x, y) for x, y in zip(a[3], b[3]))
