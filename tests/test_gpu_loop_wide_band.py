"""An iterate whose one pass takes longer than the 4 s that the one-launch loop's barriers wait (a band of 2001
entries a row at p = 36 864, FP64) runs in the chain of kernels: no timeout."""
import pytest

pytestmark = pytest.mark.gpu


def test_long_pass_is_no_timeout(lib):
    import torch

    p, half = 36864, 1000
    X = torch.randn((64, p), device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(1))
    i = torch.arange(p, device="cuda")
    lo, hi = (i - half).clamp(min=0), (i + half).clamp(max=p - 1)
    rp = torch.zeros(p + 1, device="cuda", dtype=torch.int64)
    rp[1:] = torch.cumsum(hi - lo + 1, 0)
    nnz = int(rp[-1])
    row = torch.repeat_interleave(i, hi - lo + 1)
    col = torch.arange(nnz, device="cuda") - rp[row] + lo[row]
    val = torch.where((row + col) % 3 == 0, -1e-3, 1e-3).to(torch.float64)
    val[row == col] = 1.0
    torch.cuda.synchronize()
    with lib.Solver(X, 1.0, 0.1, value_dtype=lib.F64, precision=lib.PREC_FP64, capacity=80_000_000) as s:
        s.set_omega_device(rp, col.to(torch.int32), val)
        st = s.iterate(1)
        assert st.iterations == 1
        # the step's threshold takes every entry off the diagonal
        assert st.nnz == p
