"""The one-launch iteration loop (Cov, p >= 384, fused_tail 0) against the other form of
the same steps (fused_tail 1): the same entries, decisions and iterates bit for bit; F
within the grouping of its compensated partial sums."""
import numpy as np
import pytest

from workloads import hub_factor_problem, small_problem

pytestmark = pytest.mark.gpu


def _solve(lib, X, lam1, lam2=0.1, k=None, tuning=None, **opt):
    import torch

    with lib.Solver(torch.as_tensor(X).cuda(), lam1, lam2, **opt) as s:
        if tuning:
            s.set_tuning(**tuning)
        st = s.solve() if k is None else s.iterate(k)
        return s.get_omega(), st.as_dict(), s.candidates()


def _same(a, b):
    (oa, sa, ca), (ob, sb, cb) = a, b
    for key in ("iterations", "ls_trials", "nnz", "status", "accepted_halvings", "candidates"):
        assert sa[key] == sb[key], key
    assert np.array_equal(oa.row_ptr, ob.row_ptr) and np.array_equal(oa.col, ob.col)
    assert np.array_equal(oa.val, ob.val)
    assert sa["F"] == pytest.approx(sb["F"], rel=1e-11)
    for x, y in zip(ca, cb):
        assert np.array_equal(x, y)


def _opt(lib, f64, **kw):
    return dict(value_dtype=lib.F64, precision=lib.PREC_FP64, eps=1e-9, max_iter=20000, **kw) if f64 else \
        dict(precision=lib.PREC_FP32, eps=1e-7, max_iter=20000, **kw)


@pytest.mark.parametrize("p,n,degree,lam1,f64", [
    (384, 200, 4.0, 0.15, False),       # the smallest size of the loop; 3 column blocks
    (449, 200, 4.0, 0.12, True),        # FP64, 8 blocks of 64 columns
    (500, 240, 3.0, 0.10, True),
    (1001, 400, 5.0, 0.09, False),      # 8 column blocks, the last one ragged: group maxima
    (1217, 500, 5.0, 0.08, False),      # 10 blocks, 9 rows per block of the grid
    (1600, 300, 8.0, 0.11, False),      # rows with more than 32 slots
])
def test_loop_gives_the_chains_iterates(lib, p, n, degree, lam1, f64):
    X = small_problem(p, n, degree, seed=p).astype(np.float64 if f64 else np.float32)
    other = _solve(lib, X, lam1, tuning=dict(fused_tail=1), **_opt(lib, f64))
    loop = _solve(lib, X, lam1, **_opt(lib, f64))
    _same(loop, other)
    assert loop[1]["kernel_launches"] < other[1]["kernel_launches"]
    host = _solve(lib, X, lam1, **_opt(lib, f64, device_loop=0))
    _same(loop, host)
    assert host[1]["F"] == loop[1]["F"] and host[1]["rel_change"] == loop[1]["rel_change"]


def test_loop_without_bounds_and_many_rows(lib):
    """iid X at p = 9000 (60 rows per block): 12 iterations with and without the bounds."""
    X = np.random.default_rng(21).standard_normal((1500, 9000)).astype(np.float32)
    opt = dict(precision=lib.PREC_BF16X3)
    loop = _solve(lib, X, 0.1, k=6, **opt)
    _same(loop, _solve(lib, X, 0.1, k=6, tuning=dict(fused_tail=1), **opt))
    plain = _solve(lib, X, 0.1, k=6, tuning=dict(screen_bounds=0), **opt)
    _same(loop, plain)
    assert plain[1]["F"] == loop[1]["F"]


@pytest.mark.parametrize("device_loop", [1, 0])
def test_full_bucket_leaves_the_rest_to_the_chain(lib, device_loop):
    """A hub row collects more candidates than a bucket holds."""
    X = hub_factor_problem(700, 500, 3).astype(np.float32)
    opt = dict(precision=lib.PREC_FP32, eps=1e-6, max_iter=400, device_loop=device_loop)
    loop = _solve(lib, X, 0.35, **opt)
    _same(loop, _solve(lib, X, 0.35, tuning=dict(fused_tail=1), **opt))
    assert loop[1]["candidates"] > 2 * 700


def test_loop_grows_the_candidate_capacity(lib):
    X = small_problem(512, 200, 6.0, seed=5).astype(np.float32)
    opt = dict(precision=lib.PREC_FP32, eps=1e-6, capacity=520)
    for loop in (1, 0):
        got = _solve(lib, X, 0.08, device_loop=loop, **opt)
        _same(got, _solve(lib, X, 0.08, tuning=dict(fused_tail=1), **opt))
        assert got[1]["capacity_regrows"] >= 1


def test_path_and_set_lambda_in_the_loop(lib):
    import torch

    X = torch.as_tensor(small_problem(640, 300, 4.0, 31).astype(np.float32)).cuda()
    grid = np.logspace(np.log10(0.5), np.log10(0.07), 7)
    out = []
    for form in (0, 1):
        with lib.Solver(X, grid[0], 0.1, eps=1e-7, max_iter=20000) as s:
            s.set_tuning(fused_tail=form)
            out.append(s.solve_path(grid, 0.1))
    (pa, ea), (pb, eb) = out
    for t in range(len(grid)):
        for key in ("status", "iterations", "ls_trials", "nnz"):
            assert pa[t][key] == pb[t][key], (t, key)
        assert np.array_equal(ea[t].row_ptr, eb[t].row_ptr) and np.array_equal(ea[t].val, eb[t].val)
        assert pa[t]["F"] == pytest.approx(pb[t]["F"], rel=1e-11)


def test_loop_reports_nan_and_line_search_failure(lib):
    import torch

    X = small_problem(400, 200, 4.0, 2).astype(np.float32)
    with lib.Solver(torch.as_tensor(X).cuda(), 0.1, 0.1, precision=lib.PREC_FP32, max_halvings=0) as s:
        with pytest.raises(lib.HpcError) as e:
            s.solve()
        assert e.value.status == lib.ERR_LS_FAIL
    X[3, 5] = np.nan
    with lib.Solver(torch.as_tensor(X).cuda(), 0.1, 0.1, precision=lib.PREC_FP32) as s:
        with pytest.raises(lib.HpcError) as e:
            s.solve()
        assert e.value.status == lib.ERR_NAN
