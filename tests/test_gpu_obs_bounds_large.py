"""The Obs pass over the block pairs that its bounds keep, at sizes that hold bounds (4096 pairs of
128-row blocks, p of about 11 500, and more): at every iterate the candidates and the next iterate of
a handle that has kept its bounds since its load are, bit for bit, those of a handle that loads the
data anew, sets the iterate and so takes every pair."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _x(p, n, seed):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, p), device="cuda", generator=g)
    x[:, 1:] += 0.5 * x[:, :-1].clone()
    return x


@pytest.mark.parametrize("p,n,lam1,prec,tuning", [
    (11700, 100, 0.5, "PREC_FP32", {}),       # 92 blocks, the last one ragged: 4278 pairs
    (12001, 65, 0.6, "PREC_FP32", {}),        # one sample past a K stage
    (11700, 130, 0.45, "PREC_TF32", {}),
    (12001, 300, 0.3, "PREC_FP32", dict(gram_chunk=64, gram_lead=64)),      # five chunks
    (11777, 70, 0.6, "PREC_TF32", dict(gram_chunk=32, gram_lead=32)),       # three chunks, a stage of padding left out
])
def test_kept_bounds_change_nothing(lib, p, n, lam1, prec, tuning):
    X = _x(p, n, seed=p + n)
    opt = dict(variant=lib.OBS, precision=getattr(lib, prec))
    with lib.Solver(X, lam1, 0.1, **opt) as a, lib.Solver(X, lam1, 0.1, **opt) as b:
        a.set_tuning(**tuning)
        b.set_tuning(**tuning)
        off = 0
        for step in range(10):
            if step == 6:       # another lambda1: pairs that were left out come back
                a.set_lambda(0.8 * lam1, 0.1)
                b.set_lambda(0.8 * lam1, 0.1)
            if step == 8:       # another iterate than the last pass's
                d = lib.Csr(np.arange(p + 1), np.arange(p, dtype=np.int32), np.linspace(0.5, 1.5, p))
                a.set_omega(d)
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
            off = max(off, oa.col.size - p)
        assert off > p // 10       # there is support beside the diagonal


def test_cleared_pairs_are_left_out(lib):
    """17 766 pairs at p = 24 000 and a lambda1 that nothing off the diagonal reaches: a pass takes 188
    of them, one right after a load all."""
    p = 24000
    X = _x(p, 100, seed=1)
    with lib.Solver(X, 5.0, 0.1, variant=lib.OBS) as s:
        every, kept = [], []
        for _ in range(3):
            s.load_x(X)
            every.append(s.iterate(1).ms_grad_pass)
            s.iterate(4)
            kept.append(s.iterate(1).ms_grad_pass)
    assert min(kept) < 0.5 * min(every), (kept, every)
