"""The work whose speed this project measures, through its public entry points.

Every case is a call that a user's program makes: a Gram matrix, a solve from a data
load to the estimate, a regularisation path, a batch of problems, the gradients of the
smooth loss, a tuning step.  Sizes are those of the project's workloads, tests and
benchmark rows, with ragged ones between them.

A case is a dict of plain values; ``kind`` says which call it is:

* ``gram``      S = X^T X / n into the caller's buffer (``gram``);
* ``solve``     ``load_x``, ``solve`` and the estimate into the caller's device buffers;
* ``path``      ``load_x`` and ``solve_path`` over a log-spaced lambda1 grid, estimates
                back on the host in the caller's arrays;
* ``batch``     ``load_x`` of every problem, one ``solve_batch``, every estimate;
* ``backward``  dL/dOmega (dense) and dL/dX at a given estimate (``backward``);
* ``tune``      an autograd step of the smooth loss in its sparse form, the held-out
                loss and the hypergradient at a given estimate.

Inputs follow the workloads' law: rows of X are N(0, Omega0^-1) for a sparse, strictly
diagonally dominant Omega0, drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

import paper_1710_10769_gb300 as hpc
from workloads import omega0_banded, omega0_random, omega0_tridiagonal, sample_factor

DTYPES = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}
XDTYPES = {"f32": hpc.F32, "f64": hpc.F64, "bf16": hpc.BF16}
PRECISIONS = {"auto": hpc.PREC_AUTO, "fp32": hpc.PREC_FP32, "fp64": hpc.PREC_FP64, "tf32": hpc.PREC_TF32}


def listed():
    return [
        # the smallest call: a Gram whose launches and host work cost more than its arithmetic
        dict(name="gram_f32_p300", kind="gram", p=300, n=200, x="f32", precision="auto", graph="random", degree=4.0),
        # the plain FP32 Gram (no tensor cores) at a ragged size
        dict(name="gram_plain_p3001", kind="gram", p=3001, n=1500, x="f32", precision="fp32", graph="random",
             degree=5.0),
        # the tensor-core Gram of BF16 data, whole S returned
        dict(name="gram_bf16_p16384", kind="gram", p=16384, n=8192, x="bf16", precision="auto", graph="random",
             degree=5.0),
        # FP64 throughout, the smallest workload: the iterations' latency
        dict(name="solve_f64_p500", kind="solve", p=500, n=250, x="f64", variant="cov", graph="tridiagonal",
             degree=2.0, lambda1=0.3, lambda2=0.2, host=False),
        # a small FP32 problem of odd size
        dict(name="solve_f32_p1001", kind="solve", p=1001, n=500, x="f32", variant="cov", graph="banded", degree=3.0,
             lambda1=0.15, lambda2=0.1, host=False),
        # the FP32 workload, X arriving from page-locked host memory
        dict(name="solve_f32_p16384", kind="solve", p=16384, n=8192, x="f32", variant="cov", graph="random",
             degree=5.0, lambda1=0.2, lambda2=0.1, host=True),
        # the headline workload: BF16 data at p = 65536
        dict(name="solve_bf16_p65536", kind="solve", p=65536, n=32768, x="bf16", variant="cov", graph="random",
             degree=8.0, lambda1=0.15, lambda2=0.05, host=False),
        # the Obs variant where p is far above n and S is never formed: a chain graph
        dict(name="solve_obs_p40000", kind="solve", p=40000, n=100, x="f32", variant="obs", graph="banded",
             degree=1.0, lambda1=0.46, lambda2=0.1, host=False),
        # a warm-started grid of 32 lambda1 for model selection
        dict(name="path_p8192", kind="path", p=8192, n=4096, x="f32", graph="random", degree=5.0, points=32,
             lambda1=0.8, lambda1_last=0.05, lambda2=0.1),
        # sixteen independent problems of uneven size, p = 1024 .. 16384
        dict(name="batch_16", kind="batch", p=16384, count=16, x="f32", graph="banded", degree=3.0, lambda1=0.15,
             lambda2=0.1),
        # both gradients of the smooth loss, dense dL/dOmega
        dict(name="backward_p16384", kind="backward", p=16384, n=4096, x="f32", graph="random", degree=5.0, keep=0.15,
             lambda1=0.2, lambda2=0.1),
        # one step of tuning lambda on held-out data
        dict(name="tune_p16384", kind="tune", p=16384, n=4096, nval=2048, x="f32", graph="random", degree=5.0,
             keep=0.15, lambda1=0.2, lambda2=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lambda1(rng, p, n):
    """A lambda1 above the noise level of S's off-diagonal entries, as model selection ends up with."""
    return round(max(0.1, 1.1 * math.sqrt(2.0 * math.log(max(p, 2)) / n)) * rng.uniform(1.0, 1.8), 4)


def draw(rng):
    kind = rng.choice(["gram", "solve", "solve", "obs", "path", "batch", "backward", "tune"])
    graph = rng.choice(["random", "banded"])
    degree = float(rng.randint(3, 8)) if graph == "random" else float(rng.randint(1, 3))
    if kind == "gram":
        x, precision, pmax, nmax = rng.choice([("f32", "auto", 16384, 8192), ("bf16", "auto", 16384, 8192),
                                               ("f32", "tf32", 16384, 8192), ("f32", "fp32", 6000, 3000),
                                               ("f64", "fp64", 1500, 1000)])
        return dict(kind="gram", p=_log(rng, 60, pmax), n=_log(rng, 40, nmax), x=x, precision=precision, graph=graph,
                    degree=degree)
    if kind == "solve":
        x = rng.choice(["f32", "f32", "bf16", "bf16", "f64"])
        p = _log(rng, 100, 800 if x == "f64" else 30000)
        n = max(40, int(p * rng.uniform(0.3, 0.8)))
        return dict(kind="solve", p=p, n=n, x=x, variant="cov", graph=graph, degree=degree,
                    lambda1=_lambda1(rng, p, n), lambda2=round(rng.uniform(0.05, 0.2), 3), host=rng.random() < 0.3)
    if kind == "obs":
        p, n = _log(rng, 1500, 24000), _log(rng, 80, 130)
        return dict(kind="solve", p=p, n=n, x="f32", variant="obs", graph="banded", degree=1.0,
                    lambda1=round(math.sqrt(2.0 * math.log(p) / n) * rng.uniform(1.1, 1.3), 4), lambda2=0.1, host=False)
    if kind == "path":
        p = _log(rng, 300, 8192)
        n = max(100, p // 2 + rng.randint(-p // 8, p // 8))
        last = max(0.05, 0.6 * math.sqrt(2.0 * math.log(p) / n))
        return dict(kind="path", p=p, n=n, x=rng.choice(["f32", "bf16"]), graph=graph, degree=degree,
                    points=rng.randint(6, 24), lambda1=0.8, lambda1_last=round(last, 4), lambda2=0.1)
    if kind == "batch":
        return dict(kind="batch", p=_log(rng, 600, 16384), count=rng.randint(3, 16), x="f32", graph=graph,
                    degree=degree, lambda1=0.15, lambda2=0.1)
    p = _log(rng, 300, 16384)
    n = max(64, int(p * rng.uniform(0.2, 0.6)))
    c = dict(kind=kind, p=p, n=n, x=rng.choice(["f32", "bf16"]), graph=graph, degree=degree,
             keep=round(rng.uniform(0.1, 0.6), 2), lambda1=0.2, lambda2=0.1)
    if kind == "tune":
        c["nval"] = max(32, n // 2)
    return c


# ---------------------------------------------------------------- inputs
def _graph(case, p, seed):
    if case["graph"] == "tridiagonal":
        return omega0_tridiagonal(p)
    if case["graph"] == "banded":
        return omega0_banded(p, int(case["degree"]), seed)
    return omega0_random(p, case["degree"], seed)


def _csr(a, dtype):
    t = torch.sparse_csr_tensor(torch.as_tensor(a.indptr.astype(np.int64)), torch.as_tensor(a.indices.astype(np.int64)),
                                torch.as_tensor(a.data), size=a.shape)
    return t.to("cuda", dtype)


def _samples(omega0, n, seed, stream, dtype):
    """n rows of N(0, Omega0^-1): x = Omega0^-1 B^T z with Omega0 = B^T B, by Chebyshev iteration on
    the Jacobi-scaled matrix, whose eigenvalues lie within 1 +- rho (Gershgorin)."""
    f = sample_factor(omega0)
    p = f.p
    work = torch.float64 if dtype == torch.float64 else torch.float32
    bt, om = _csr(f.Bt, work), _csr(f.omega, work)
    d = torch.as_tensor(f.diag, device="cuda").to(work)[:, None]
    rho = float(np.max((np.asarray(abs(f.omega).sum(axis=1)).ravel() - f.diag) / f.diag))
    steps = 40 if work == torch.float64 else 20
    gen = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)
    out = torch.empty((n, p), dtype=dtype, device="cuda")
    for r0 in range(0, n, 2048):
        c = min(n, r0 + 2048) - r0
        b = bt @ torch.randn((f.m, c), dtype=work, device="cuda", generator=gen)
        x = b / d
        if rho > 0.0:
            res = (b - om @ x) / d
            step, gamma = res.clone(), rho
            for _ in range(steps):
                x += step
                res -= (om @ step) / d
                new = 1.0 / (2.0 / rho - gamma)
                step = (new * gamma) * step + (2.0 * new / rho) * res
                gamma = new
        out[r0:r0 + c] = x.t()
    return out


def _estimate(omega0, keep, seed):
    """An estimate of Omega0 as a solve leaves it: the diagonal and a share of the edges, shrunk;
    (row_ptr, col, val) on the host."""
    a = omega0.tocoo()
    up = a.row < a.col
    i, j, v = a.row[up], a.col[up], a.data[up]
    rng = np.random.Generator(np.random.PCG64(seed + 17))
    sel = rng.permutation(i.size)[:max(1, round(keep * i.size))]
    i, j, v = i[sel], j[sel], v[sel] * 0.4
    dg = np.arange(omega0.shape[0])
    row, col = np.concatenate([dg, i, j]), np.concatenate([dg, j, i])
    val = np.concatenate([omega0.diagonal() * 0.8, v, v])
    order = np.lexsort((col, row))
    row_ptr = np.zeros(omega0.shape[0] + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(row, minlength=omega0.shape[0]))
    return hpc.Csr(row_ptr, col[order].astype(np.int32), val[order].astype(np.float32).astype(np.float64))


def _batch_sizes(case):
    k = case["count"]
    return [max(64, case["p"] * (t + 1) // k) for t in range(k)]


def _solver(case, n, p, stream=None):
    opt = dict(value_dtype=hpc.F64) if case["x"] == "f64" else {}
    variant = hpc.OBS if case.get("variant") == "obs" else hpc.COV
    return hpc.Solver(None, case["lambda1"], case["lambda2"], variant=variant, stream=stream, n=n, p=p,
                      xdtype=XDTYPES[case["x"]], **opt)


# entries of an estimate that the caller's buffers have room for, per row
ROOM = 24


def _buffers(case, p):
    wide = torch.float64 if case["x"] == "f64" else torch.float32
    return {"row_ptr": torch.zeros(p + 1, dtype=torch.int64, device="cuda"),
            "col": torch.zeros(ROOM * p, dtype=torch.int32, device="cuda"),
            "val": torch.zeros(ROOM * p, dtype=wide, device="cuda")}


def _grid(case):
    return np.geomspace(case["lambda1"], case["lambda1_last"], case["points"])


def prepare(case, seed):
    kind, dtype = case["kind"], DTYPES[case["x"]]
    if kind == "batch":
        state = dict(case=case, X=[], solvers=[], buffers=[])
        for t, p in enumerate(_batch_sizes(case)):
            n = max(32, p // 2)
            state["X"].append(_samples(_graph(case, p, 100 * seed + t), n, 100 * seed + t, 0, dtype))
            state["solvers"].append(_solver(case, n, p, torch.cuda.Stream()))
            state["buffers"].append(_buffers(case, p))
        torch.cuda.synchronize()
        return state
    p, n = case["p"], case["n"]
    omega0 = _graph(case, p, seed)
    X = _samples(omega0, n, seed, 0, dtype)
    if kind == "gram":
        wide = torch.float64 if case["precision"] == "fp64" else torch.float32
        return dict(case=case, X=X, S=torch.empty((p, p), dtype=wide, device="cuda"))
    state = dict(case=case, X=X, solver=_solver(case, n, p))
    if kind == "solve":
        state["buffers"] = _buffers(case, p)
    if kind == "path":
        cap = ROOM * p * case["points"]
        state["arrays"] = (np.zeros(case["points"] * (p + 1), np.int64), np.zeros(cap, np.int32),
                           np.zeros(cap, np.float32))
    if kind == "solve" and case["host"]:
        state["X"] = torch.empty(X.shape, dtype=dtype, pin_memory=True).copy_(X)
    if kind in ("backward", "tune"):
        state["solver"].load_x(X)
        est = _estimate(omega0, case["keep"], seed)
        state["solver"].set_omega(est)
        state["omega"] = torch.as_tensor(est.val).to("cuda", torch.float32)
    if kind == "tune":
        state["Xval"] = _samples(omega0, case["nval"], seed, 1, dtype)
    torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------- one pass
def _result(solver, buffers):
    solver.get_omega_device(buffers["row_ptr"], buffers["col"], buffers["val"])
    return buffers


def run(state):
    case = state["case"]
    kind, X = case["kind"], state["X"]
    if kind == "gram":
        hpc.gram(X, state["S"], precision=PRECISIONS[case["precision"]])
        return state["S"]
    if kind == "batch":
        for solver, x in zip(state["solvers"], X):
            solver.load_x(x)
        stats = hpc.solve_batch(state["solvers"])
        return {"F": [s["F"] for s in stats], "omega": [_result(s, b) for s, b in zip(state["solvers"], state["buffers"])]}
    solver = state["solver"]
    if kind == "solve":
        solver.load_x(X)
        stats = solver.solve()
        return {"F": stats.F, **_result(solver, state["buffers"])}
    if kind == "path":
        solver.load_x(X)
        points, estimates = solver.solve_path(_grid(case), case["lambda2"])
        row_ptr, col, val = state["arrays"]
        np.concatenate([e.row_ptr for e in estimates], out=row_ptr)
        used = sum(e.col.size for e in estimates)
        np.concatenate([e.col for e in estimates], out=col[:used])
        np.concatenate([e.val for e in estimates], out=val[:used], casting="same_kind")
        return {"F": [q["F"] for q in points], "row_ptr": row_ptr, "col": col, "val": val}
    if kind == "backward":
        d_omega, d_x = solver.backward(X)
        return {"d_omega": d_omega, "d_x": d_x}
    x = X.detach().requires_grad_()
    omega = state["omega"].detach().requires_grad_()
    loss = hpc.concord_smooth_loss(x, omega, solver)
    loss.backward()
    held = solver.heldout_loss(state["Xval"])
    d1, d2, _ = solver.hypergrad(state["Xval"])
    return {"loss": loss.detach(), "d_x": x.grad, "d_omega": omega.grad, "heldout": held, "d_lambda1": d1,
            "d_lambda2": d2}


# ---------------------------------------------------------------- the work a pass cannot do without
def work(case):
    kind, es = case["kind"], {"f32": 4, "f64": 8, "bf16": 2}[case["x"]]
    vs = 8 if case["x"] == "f64" else 4
    if kind == "batch":
        sizes = [(p, max(32, p // 2)) for p in _batch_sizes(case)]
        return {"bytes": sum(n * p * es + 16 * p for p, n in sizes), "flops": sum(n * p * (p + 1.0) for p, n in sizes)}
    p, n = case["p"], case["n"]
    x = n * p * es
    if kind == "gram":
        return {"bytes": x + p * p * (8 if case["precision"] == "fp64" else 4), "flops": n * p * (p + 1.0)}
    if kind == "solve" and case["variant"] == "obs":
        return {"bytes": x + 16 * p, "flops": 2.0 * n * p * p}     # one product Z = YX / n
    if kind in ("solve", "path"):
        # the Gram, and the estimate (a diagonal at least) written per point
        return {"bytes": x + (8 + 4 + vs) * p * case.get("points", 1), "flops": n * p * (p + 1.0)}
    nnz = p * (1 + case["keep"] * case["degree"] * (1 if case["graph"] == "random" else 2))
    if kind == "backward":
        # S's upper triangle read, dL/dOmega written; X read, dL/dX written
        return {"bytes": 2 * p * (p + 1) + 4 * p * p + x + 4 * n * p, "flops": 4.0 * nnz * n + 2.0 * nnz * p}
    # X and X_val read, dL/dX written, the support's values and S entries
    return {"bytes": x + 4 * n * p + case["nval"] * p * es + 40 * nnz, "flops": 4.0 * nnz * n + 2.0 * nnz * case["nval"]}


# ---------------------------------------------------------------- the same in 64 bits
def _gram64(X):
    n, p = X.shape
    S = torch.empty((p, p), dtype=torch.float64, device="cuda")
    Xd = X.cuda().double()
    for j in range(0, p, 4096):
        S[:, j:j + 4096] = Xd.t() @ Xd[:, j:j + 4096]
    return S / n


def _solve64(S, lam1, lam2, omega, eps=1e-6, max_iter=1000):
    """Proximal gradient with backtracking in dense FP64 from the iterate omega."""
    eye = torch.eye(S.shape[0], dtype=torch.bool, device=S.device)
    for _ in range(max_iter):
        W = omega @ S
        dg = omega.diagonal()
        G = 0.5 * (W + W.t()) + lam2 * omega - torch.diag(1.0 / dg)
        tau = 1.0
        while True:
            z = omega - tau * G
            new = torch.where(eye, z, torch.sign(z) * (z.abs() - tau * lam1).clamp(min=0.0))
            nd = new.diagonal()
            if bool((nd > 0).all()):
                D = new - omega
                n2 = (D * D).sum()
                r = D.diagonal() / dg
                if bool(0.5 * ((D @ S) * D).sum() + 0.5 * lam2 * n2 + (r - torch.log1p(r)).sum() <= n2 / (2 * tau)):
                    break
            tau *= 0.5
        rel = float(n2.sqrt() / omega.norm())
        F = -dg.log().sum() + 0.5 * (W * omega).sum() + 0.5 * lam2 * (omega * omega).sum() + lam1 * (
            omega.abs().sum() - dg.sum())
        omega = new
        if rel < eps:
            break
    return omega, float(F)


def _nonzeros(omegas, room):
    """The values of the estimates one after another, in a buffer of the size that run() fills."""
    out = torch.zeros(room, dtype=omegas[0].dtype, device="cuda")
    at = 0
    for omega in omegas:
        v = omega[(omega != 0) | torch.eye(omega.shape[0], dtype=torch.bool, device="cuda")]
        out[at:at + v.numel()] = v
        at += v.numel()
    return out


def _mm(est, values, dense):
    p = est.row_ptr.size - 1
    a = torch.sparse_csr_tensor(torch.as_tensor(est.row_ptr).cuda(), torch.as_tensor(est.col.astype(np.int64)).cuda(),
                                values, size=(p, p))
    return a @ dense


def exact(case, seed):
    kind = case["kind"]
    small = case["p"] <= 1200
    if kind == "batch" or (kind in ("solve", "path") and not small):
        return None
    dtype = DTYPES[case["x"]]
    omega0 = _graph(case, case["p"], seed)
    X = _samples(omega0, case["n"], seed, 0, dtype)
    S = _gram64(X)
    if kind == "gram":
        return S
    if kind == "solve":
        omega, F = _solve64(S, case["lambda1"], case["lambda2"], torch.eye(case["p"], dtype=S.dtype, device="cuda"))
        return {"F": F, "row_ptr": None, "col": None, "val": _nonzeros([omega], ROOM * case["p"])}
    if kind == "path":
        omega, omegas, Fs = torch.eye(case["p"], dtype=S.dtype, device="cuda"), [], []
        for lam in _grid(case):
            omega, F = _solve64(S, float(lam), case["lambda2"], omega)
            omegas.append(omega)
            Fs.append(F)
        return {"F": Fs, "row_ptr": None, "col": None,
                "val": _nonzeros(omegas, ROOM * case["p"] * case["points"])}
    est = _estimate(omega0, case["keep"], seed)
    p, n, lam2 = case["p"], case["n"], case["lambda2"]
    row = torch.as_tensor(np.repeat(np.arange(p), np.diff(est.row_ptr))).cuda()
    col = torch.as_tensor(est.col.astype(np.int64)).cuda()
    w = torch.as_tensor(est.val).cuda()
    diag = row == col
    d_x = _mm(est, w, _mm(est, w, X.double().t().contiguous())).t() / n
    if kind == "backward":
        OS = _mm(est, w, S)
        G = 0.5 * (OS + OS.t())
        del OS
        G[row, col] += lam2 * w - torch.where(diag, 1.0 / w, torch.zeros_like(w))
        return {"d_omega": G, "d_x": d_x}
    sym = lambda T: 0.5 * (T[row, col] + T[col, row])  # noqa: E731
    T = _mm(est, w, S)
    g = sym(T) + lam2 * w - torch.where(diag, 1.0 / w, torch.zeros_like(w))
    log = w[diag].log().sum()
    loss = -log + 0.5 * (w * T[row, col]).sum() + 0.5 * lam2 * (w * w).sum()
    Tv = _mm(est, w, _gram64(_samples(omega0, case["nval"], seed, 1, dtype)))
    held = -log + 0.5 * (w * Tv[row, col]).sum()
    b = sym(Tv) - torch.where(diag, 1.0 / w, torch.zeros_like(w))
    del T, Tv
    hess = lambda v: sym(_mm(est, v, S)) + lam2 * v + torch.where(diag, v / (w * w), torch.zeros_like(v))  # noqa: E731
    v, r = torch.zeros_like(b), b.clone()
    q, rr = r.clone(), (r * r).sum()
    stop = 1e-24 * float(rr)
    for _ in range(400):
        Aq = hess(q)
        a = rr / (q * Aq).sum()
        v += a * q
        r -= a * Aq
        new = (r * r).sum()
        if float(new) <= stop:
            break
        q = r + (new / rr) * q
        rr = new
    off = torch.where(diag, torch.zeros_like(w), torch.sign(w))
    return {"loss": loss, "d_x": d_x, "d_omega": g, "heldout": float(held), "d_lambda1": -float((v * off).sum()),
            "d_lambda2": -float((v * w).sum())}
