"""hpc_set_omega with on_device = 1 from memory that its kernels cannot or may not read: arrays off their
elements' alignment and host arrays come by copies, an allocation that is too short is an error."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = 64


def _csr():
    v = np.linspace(1.0, 2.0, P)
    return np.arange(P + 1, dtype=np.int64), np.arange(P, dtype=np.int32), v


def _set(lib, s, ptrs):
    return lib.load().hpc_set_omega(s._h, P, *(C.c_void_p(q) for q in ptrs), lib.F64, 1)


@pytest.mark.parametrize("kind", ["aligned", "misaligned", "pinned"])
def test_taken(lib, kind):
    import torch

    arrays = _csr()
    if kind == "pinned":
        keep = [torch.as_tensor(a).pin_memory() for a in arrays]
        ptrs = [t.data_ptr() for t in keep]
    else:
        keep, ptrs = [], []
        for a in arrays:
            off = a.itemsize // 2 if kind == "misaligned" else 0
            t = torch.zeros(a.nbytes + 16, dtype=torch.uint8, device="cuda")
            t[off:off + a.nbytes] = torch.as_tensor(a.view(np.uint8)).cuda()
            keep.append(t)
            ptrs.append(t.data_ptr() + off)
    torch.cuda.synchronize()
    with lib.Solver(torch.randn(100, P, device="cuda"), 0.2, 0.1) as s:
        assert _set(lib, s, ptrs) == lib.OK
        got = s.get_omega()
        assert np.array_equal(got.col, arrays[1]) and np.array_equal(got.val, arrays[2].astype(np.float32))


def test_short_allocation_is_an_error(lib):
    import torch

    rt = C.CDLL("libcudart.so.13")
    q = C.c_void_p()
    with lib.Solver(torch.randn(100, P, device="cuda"), 0.2, 0.1) as s:
        assert rt.cudaMalloc(C.byref(q), C.c_size_t(256)) == 0
        keep = [torch.as_tensor(a).cuda() for a in _csr()[1:]]
        torch.cuda.synchronize()
        assert _set(lib, s, [q.value] + [t.data_ptr() for t in keep]) == lib.ERR_CUDA
        assert s.get_omega().col.size == P         # the iterate is as it was
        assert rt.cudaFree(q) == 0
