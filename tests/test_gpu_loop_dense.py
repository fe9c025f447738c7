"""Where the one-launch loop (Cov) leaves an iteration to the chain of kernels: dense iterates, hub rows,
no bounds.  The same entries, decisions and iterates as with fused_tail 1, and the count of launches
tells which form ran."""
import numpy as np
import pytest

from workloads import hub_factor_problem, small_problem

pytestmark = pytest.mark.gpu


def _run(lib, X, lam1, k, f64=False, tuning=None, **opt):
    import torch

    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64, **opt) if f64 else dict(precision=lib.PREC_FP32, **opt)
    with lib.Solver(torch.as_tensor(X).cuda(), lam1, 0.1, **opt) as s:
        s.set_tuning(**(tuning or {}))
        st = s.iterate(k).as_dict()
        return s.get_omega(), st, s.candidates()


def _same(a, b):
    (oa, sa, ca), (ob, sb, cb) = a, b
    for key in ("iterations", "ls_trials", "nnz", "status", "accepted_halvings", "candidates"):
        assert sa[key] == sb[key], key
    assert np.array_equal(oa.row_ptr, ob.row_ptr) and np.array_equal(oa.col, ob.col)
    assert np.array_equal(oa.val, ob.val)
    assert sa["F"] == pytest.approx(sb["F"], rel=1e-11)
    for x, y in zip(ca, cb):
        assert np.array_equal(x, y)


def _x(p, n, f64=False):
    x = np.random.default_rng(p).standard_normal((n, p))
    x[:, 1:] += 0.4 * x[:, :-1]
    return x.astype(np.float64 if f64 else np.float32)


@pytest.mark.parametrize("loop", [1, 0])
@pytest.mark.parametrize("case", ["rows_of_1500", "rows_of_90", "fp64", "hub", "no_bounds"])
def test_dense_iterations_run_in_the_chain(lib, case, loop):
    tuning, f64 = {}, case == "fp64"
    if case == "rows_of_1500":
        X, lam1, k = _x(2000, 300), 0.02, 3             # buckets and pages overflow
    elif case == "rows_of_90":
        X, lam1, k = _x(2000, 300), 0.1, 8              # terms of the tasks
    elif case == "fp64":
        X, lam1, k = _x(1000, 300, True), 0.05, 4
    elif case == "hub":
        X, lam1, k = hub_factor_problem(1500, 500, 3).astype(np.float32), 0.35, 8      # one row's support
    else:
        X, lam1, k, tuning = _x(10000, 300), 0.4, 4, dict(screen_bounds=0)
    got = _run(lib, X, lam1, k, f64, tuning, device_loop=loop)
    _same(got, _run(lib, X, lam1, k, f64, dict(fused_tail=1, **tuning), device_loop=loop))
    assert got[1]["kernel_launches"] > 20


@pytest.mark.parametrize("p,n,lam1,f64", [(600, 400, 0.15, False), (609, 400, 0.15, False), (1216, 500, 0.15, False),
                                          (1217, 500, 0.15, False), (900, 400, 0.15, True)])
def test_light_iterations_stay_in_the_loop(lib, p, n, lam1, f64):
    """Also the edges of the grid's rule (76 SMs' blocks of up to 16 rows, then one per SM)."""
    X = small_problem(p, n, 4.0, seed=p).astype(np.float64 if f64 else np.float32)
    om, st, _ = _run(lib, X, lam1, 30, f64)
    other = _run(lib, X, lam1, 30, f64, dict(fused_tail=1))
    assert np.array_equal(om.row_ptr, other[0].row_ptr) and np.array_equal(om.val, other[0].val)
    assert st["F"] == pytest.approx(other[1]["F"], rel=1e-11)
    assert st["kernel_launches"] == 2
