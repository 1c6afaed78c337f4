"""Work lists that are made on first use (owner-computes residual, tcgen05 product) and find no memory
half way leave nothing behind: the call reports HM_ERR_OOM, and once there is memory the handle
holds exactly what one holds that never failed, with the same result.
"""

import ctypes
import gc

import pytest

pytestmark = pytest.mark.gpu


class Full:
    """Takes the device's memory but for `left` pieces of 2 MB."""

    def __init__(self, left):
        import torch
        from paper_2307_03968_gb300.hm import load
        gc.collect()                                       # nothing of earlier tests is given back in between
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.rt, self.held = load(), []
        for size in (1 << 30, 64 << 20, 2 << 20, 64 << 10):
            while True:
                p = ctypes.c_void_p()
                if self.rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) != 0:
                    self.rt.cudaGetLastError()
                    break
                p.size = size
                self.held.append(p)
        for p, _ in zip([q for q in self.held if q.size == 2 << 20], range(left)):
            self.held.remove(p)
            self.rt.cudaFree(p)

    def close(self):
        while self.held:
            self.rt.cudaFree(self.held.pop())


@pytest.mark.parametrize("prod,res", [(16, 1017), (1016, 16)])
def test_failed_lists_leave_nothing(prod, res):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import icosphere
    from paper_2307_03968_gb300.hm import HMatrix, HmError, HM_ERR_OOM
    nrhs = 8
    handles = []
    for _ in range(2):
        A = HMatrix.build(*icosphere(4, 1.0), leaf_size=16, arity=8, adm=2.0, aca_tol=1e-3, levels=1)
        A.factor_leaf()
        handles.append(A)
    A, T = handles
    x = torch.randn((nrhs, A.n), dtype=torch.complex64, device="cuda")
    y, r, ref = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)

    def call(M, out):
        if res == 1017:
            M.residual(x, y, out, n_levels=1)
        else:
            M.apply(x, out, n_levels=1, fp64_accumulate=False)

    for M in handles:                                      # buffers and device code of the calls
        M.set_tuning(nrhs, 16, 16)
        M.apply(x, y, n_levels=1, fp64_accumulate=False)
        M.residual(x, y, r, n_levels=1)
        M.set_tuning(nrhs, prod, res)
    call(T, ref)
    torch.cuda.synchronize()
    held = A.info().device_bytes
    full = Full(1)
    try:
        with pytest.raises(HmError) as e:
            call(A, r)
    finally:
        full.close()
    assert e.value.status == HM_ERR_OOM
    assert A.info().device_bytes == held
    call(A, r)
    torch.cuda.synchronize()
    assert A.info().device_bytes == T.info().device_bytes
    assert ((r - ref).norm() / ref.norm()).item() < 1e-5
    for M in handles:
        M.close()
