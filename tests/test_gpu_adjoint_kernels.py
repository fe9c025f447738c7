"""The differentiation kernels at the sizes where their tilings can go wrong, against FP64: the
dense gradient's entry list and its overflow, the held-out support product's pieces and batches,
the one-launch CG in both forms, and hpc_set_omega's checks on device arrays."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


def _omega(p, degree, seed, hub=None):
    """Symmetric, positive diagonal, FP32 values; hub: a row that meets every third column."""
    rng = np.random.default_rng(seed)
    m = int(p * degree / 2)
    i, j = rng.integers(0, p, m), rng.integers(0, p, m)
    if hub is not None:
        j2 = np.arange(0, p, 3)
        i, j = np.concatenate([i, np.full(j2.size, hub)]), np.concatenate([j, j2])
    off = i != j
    a = sp.coo_matrix((rng.uniform(-0.3, 0.3, off.sum()) / max(degree, 1), (i[off], j[off])), shape=(p, p)).tocsr()
    a = ((a + a.T) * 0.5 + sp.diags(rng.uniform(0.7, 1.3, p))).tocsr()
    a.sort_indices()
    a.data = a.data.astype(np.float32).astype(np.float64)
    return a


def _csr(lib, a):
    return lib.Csr(a.indptr.astype(np.int64), a.indices.astype(np.int32), a.data)


def _solver(lib, X, f64=False, lam2=0.1):
    opt = dict(value_dtype=lib.F64, precision=lib.PREC_FP64) if f64 else dict(precision=lib.PREC_FP32)
    return lib.Solver(X, 0.1, lam2, **opt)


@pytest.mark.parametrize("p,degree,hub,f64", [
    (1, 0.0, None, False),
    (65, 3.0, None, False),        # a ragged second block
    (192, 3.0, None, False),       # whole blocks: 16-byte loads
    (256, 30.0, None, False),      # more entries than the list holds
    (321, 2.0, 320, False),        # a hub row in the last block
    (70, 4.0, 3, True),
])
def test_gradients_match_fp64(lib, p, degree, hub, f64):
    import torch

    n, lam2, u = 90, 0.1, 2.0 ** -53 if f64 else 2.0 ** -24
    X = torch.as_tensor(np.random.default_rng(p).standard_normal((n, p))).to(torch.float64 if f64 else torch.float32)
    a = _omega(p, degree, p, hub)
    with _solver(lib, X.cuda(), f64, lam2) as s:
        s.set_omega(_csr(lib, a))
        g, dx = s.backward(X.cuda())
        S = s.s_entries(np.repeat(np.arange(p), p), np.tile(np.arange(p), p)).reshape(p, p)
    A, Xd = a.toarray(), X.double().numpy()
    W = A @ S
    ref = 0.5 * (W + W.T) + lam2 * A - np.diag(1.0 / A.diagonal())
    k = int(np.diff(a.indptr).max())
    B = np.abs(A) @ np.abs(S)
    bound = (k + 4) * u * (0.5 * (B + B.T) + lam2 * np.abs(A) + np.diag(1.0 / A.diagonal()))
    assert np.all(np.abs(g.double().cpu().numpy() - ref) <= bound)
    bound = (2 * k + 5) * u * (np.abs(Xd) @ np.abs(A) @ np.abs(A)) / n
    assert np.all(np.abs(dx.double().cpu().numpy() - Xd @ A @ A / n) <= bound)


@pytest.mark.parametrize("p,nval,degree,hub,f64", [
    (40, 1, 2.0, None, False),
    (130, 33, 3.0, 7, False),      # a row of 40 entries: three batches
    (90, 2049, 3.0, None, False),  # a second piece of one sample
    (64, 4100, 2.0, 1, True),
])
def test_heldout_loss_matches_fp64(lib, p, nval, degree, hub, f64):
    import torch

    dt, u = (torch.float64, 2.0 ** -53) if f64 else (torch.float32, 2.0 ** -24)
    rng = np.random.default_rng(p + nval)
    X = torch.as_tensor(rng.standard_normal((50, p))).to(dt).cuda()
    V = torch.as_tensor(rng.standard_normal((nval, p))).to(dt)
    a = _omega(p, degree, p, hub)
    with _solver(lib, X, f64) as s:
        s.set_omega(_csr(lib, a))
        got = s.heldout_loss(V.cuda())
    A, Vd = a.toarray(), V.double().numpy()
    ref = -np.log(A.diagonal()).sum() + 0.5 * ((Vd @ A) ** 2).sum() / nval
    # chains of a row's terms and of the 16 products a thread sums in the value type
    k = int(np.diff(a.indptr).max())
    Y = np.abs(Vd) @ np.abs(A)
    assert abs(got - ref) <= (k + 18) * u * 0.5 * (Y * Y).sum() / nval + 1e-12 * (1 + abs(ref))


@pytest.mark.parametrize("p,degree,f64", [
    (60, 2.0, False),
    (700, 4.0, True),              # an entry per thread, several blocks
    (1500, 150.0, False),          # more entries than threads: the strided form
])
def test_hypergradient_matches_fp64_cg(lib, p, degree, f64):
    import torch

    lam2, dt = 0.2, torch.float64 if f64 else torch.float32
    rng = np.random.default_rng(p)
    X = torch.as_tensor(rng.standard_normal((2 * p, p))).to(dt)
    V = torch.as_tensor(rng.standard_normal((p, p))).to(dt)
    a = _omega(p, degree, p)
    with _solver(lib, X.cuda(), f64, lam2) as s:
        s.set_omega(_csr(lib, a))
        d1, d2, info = s.hypergrad(V.cuda(), tol=1e-10)
        S = s.s_entries(np.repeat(np.arange(p), p), np.tile(np.arange(p), p)).reshape(p, p)
    Vd = V.double().numpy()
    Sv = Vd.T @ Vd / V.shape[0]
    row, col = np.repeat(np.arange(p), np.diff(a.indptr)), a.indices
    dg, w = row == col, a.data
    sym = lambda T: 0.5 * (T[row, col] + T[col, row])  # noqa: E731
    mat = lambda v: sp.csr_matrix((v, a.indices, a.indptr), shape=(p, p))  # noqa: E731
    b = sym(a @ Sv) - np.where(dg, 1.0 / w, 0.0)
    hess = lambda v: sym(mat(v) @ S) + lam2 * v + np.where(dg, v / (w * w), 0.0)  # noqa: E731
    v, r = np.zeros_like(b), b.copy()
    q, rr = r.copy(), r @ r
    stop = 1e-24 * rr
    for _ in range(500):
        Aq = hess(q)
        t = rr / (q @ Aq)
        v += t * q
        r -= t * Aq
        new = r @ r
        if new <= stop:
            break
        q, rr = r + (new / rr) * q, new
    assert info["converged"] == 1 and info["support"] == a.nnz
    e1, e2 = -(v * np.where(dg, 0.0, np.sign(w))).sum(), -(v * w).sum()
    # v's error is at most (tol |b| + |b's error|) / lambda2; b's error: a row's terms and 18 roundings
    k = int(np.diff(a.indptr).max())
    db = (k + 18) * (2.0 ** -53 if f64 else 2.0 ** -24) * sym(np.abs(a) @ (np.abs(Vd).T @ np.abs(Vd)) / V.shape[0])
    err = (1e-10 * np.linalg.norm(b) + np.linalg.norm(db)) / lam2
    assert abs(d1 - e1) <= err * np.sqrt((~dg).sum() + 1) and abs(d2 - e2) <= err * np.linalg.norm(w)


def test_device_omega_is_checked_as_host_omega(lib):
    import torch

    p = 300
    X = torch.as_tensor(np.random.default_rng(1).standard_normal((50, p)).astype(np.float32)).cuda()
    a = _omega(p, 4.0, 2)
    good = [a.indptr.astype(np.int64), a.indices.astype(np.int32), a.data.copy()]
    dpos = [int(np.nonzero((a.indices == i) & (np.arange(a.nnz) >= a.indptr[i]) & (np.arange(a.nnz) < a.indptr[i + 1]))[0][0])
            for i in range(p)]

    def broken(*edits):
        g = [x.copy() for x in good]
        for which, at, value in edits:
            g[which][at] = value
        return g

    off = int(next(t for t in range(a.nnz) if t not in set(dpos)))
    cases = [good,
             broken((0, 0, 1)), broken((0, p, a.nnz - 1)), broken((0, 5, int(a.indptr[7]))),
             broken((1, off, p)), broken((1, off, -1)), broken((1, dpos[40], int(a.indices[dpos[40]]) + p)),
             broken((2, dpos[9], 0.0)), broken((2, dpos[9], np.nan)), broken((2, off, np.inf)),
             broken((2, dpos[9], -1.0), (2, off, np.nan)), broken((2, dpos[299], -1.0), (2, off, np.nan))]
    for dt in (np.float64, np.float32):
        for g in cases:
            out = []
            for device in (False, True):
                with lib.Solver(X, 0.1, 0.1, precision=lib.PREC_FP32) as s:
                    try:
                        if device:
                            s.set_omega_device(torch.as_tensor(g[0]).cuda(), torch.as_tensor(g[1]).cuda(),
                                               torch.as_tensor(g[2].astype(dt)).cuda())
                        else:
                            s.set_omega(lib.Csr(g[0], g[1], g[2]))
                        out.append(s.get_omega())
                    except lib.HpcError as e:
                        out.append(e.status)
            if isinstance(out[0], int):
                assert out[0] == out[1]
            else:
                assert all(np.array_equal(getattr(out[0], f), getattr(out[1], f)) for f in ("row_ptr", "col", "val"))
