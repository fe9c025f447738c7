"""The Obs Z product in TF32 with short accumulation chunks, at n whose last K stage of 32 holds
samples or only padding, against FP64: with Omega = I and lambda1 = 0 every entry is a
candidate with G_ij = Z_ij off the diagonal, Z = X^T X / n."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,chunk,lead", [
    (70, 32, 32),       # four stages of 32, the last all padding and a chunk of its own
    (280, 32, 0),       # ten stages in chunks of 4, 4, 1, 1: the last all padding
    (257, 96, 96),      # chunks of 3, 3, 3, 1: the same
    (300, 32, 0),       # every stage holds samples
    (40, 0, 0),         # one chunk, one sample stage and one of padding in it
])
def test_short_chunks_match_fp64(lib, n, chunk, lead):
    import torch

    p = 300
    X = np.random.default_rng(n).standard_normal((n, p)).astype(np.float32)
    with lib.Solver(None, 0.0, 0.1, variant=lib.OBS, precision=lib.PREC_TF32, n=n, p=p) as s:
        s.set_tuning(gram_chunk=chunk, gram_lead=lead)
        s.load_x(torch.as_tensor(X).cuda())
        s.iterate(1)
        r, c, _, g = s.candidates()
    assert r.size == p * p
    G = np.zeros((p, p))
    G[r, c] = g
    S = X.astype(np.float64).T @ X.astype(np.float64) / n
    off = ~np.eye(p, dtype=bool)
    # each operand is rounded by 2^-11 relative; |x_i|.|x_j| <= n sqrt(S_ii S_jj); as much again
    # for the accumulation
    tol = 2.0 ** -9 * np.sqrt(np.outer(np.diag(S), np.diag(S)))
    assert (np.abs(G - S)[off] <= tol[off]).all(), np.abs(G - S)[off].max()
