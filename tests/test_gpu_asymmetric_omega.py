"""hpc_set_omega with entries whose transpose is absent or has another value, at sizes of the one-launch
iteration loop: the same outcome (iterates, or the status of the error) as with fused_tail 1."""
import numpy as np
import pytest
import scipy.sparse as sp

from workloads import small_problem

pytestmark = pytest.mark.gpu


def _outcome(lib, X, om, f64, tail, loop):
    import torch

    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64) if f64 else dict(precision=lib.PREC_FP32)
    with lib.Solver(torch.as_tensor(X).cuda(), 0.15, 0.1, device_loop=loop, **opt) as s:
        s.set_tuning(fused_tail=tail)
        s.solve()               # a captured loop, from the identity
        s.set_omega(om)
        try:
            st = s.iterate(3).as_dict()
        except lib.HpcError as e:
            return ("error", e.status)
        got = s.get_omega()
        return (st["iterations"], st["ls_trials"], st["nnz"]), got.row_ptr, got.col, got.val


@pytest.mark.parametrize("loop", [1, 0])
@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("kind", ["one_sided_above", "one_sided_below", "other_value"])
def test_same_outcome_as_the_other_form(lib, kind, f64, loop):
    p = 400
    X = small_problem(p, 200, 4.0, 7).astype(np.float64 if f64 else np.float32)
    S = X.T.astype(np.float64) @ X / X.shape[0]
    a = np.abs(S - np.diag(np.diag(S)))
    i, j = np.unravel_index(np.argmax(a) if kind != "one_sided_below" else np.argmin(a + 9.0 * np.eye(p)), a.shape)
    D = sp.lil_matrix(np.eye(p))
    D[i, j] = 0.01
    if kind == "other_value":
        D[j, i] = 0.02
    D = sp.csr_matrix(D)
    om = lib.Csr(D.indptr.astype(np.int64), D.indices.astype(np.int32), D.data)
    a, b = _outcome(lib, X, om, f64, 0, loop), _outcome(lib, X, om, f64, 1, loop)
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y
