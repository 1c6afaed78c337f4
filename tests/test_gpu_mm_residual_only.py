"""A program that only forms residuals (hm_residual, hm_apply with FP64-class accumulation) holds no
operand streams of the FP32 product: those, twice the blocks' bytes, come with the first call that
runs a product, which then times its candidates.
"""

import pytest

from test_gpu_mm import Blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [6, 40])
def test_streams_come_with_the_first_product(nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B = Blocks(nrhs, 1.0)
    A = B.operator()
    blocks = 8 * (A.info().near_elems + sum(A.info().far_elems))
    x, _ = B.vectors(nrhs)
    xt = torch.from_numpy(x).cuda()
    y, r = torch.empty_like(xt), torch.empty_like(xt)
    A.apply(xt, y, n_levels=1)                             # FP64-class accumulation
    A.residual(y, xt, r, n_levels=1)
    held = A.info().device_bytes
    prod, res, prod_ms, res_ms = A.tuning(nrhs)
    assert prod in (8, 16) and prod_ms == 0 and res in (0, 8, 16, 1017) and res_ms > 0
    A.residual(y, xt, r, n_levels=1)
    assert A.info().device_bytes == held
    A.apply(xt, y, n_levels=1, fp64_accumulate=False)
    assert A.info().device_bytes - held >= 2 * blocks
    prod, after, prod_ms, _ = A.tuning(nrhs)
    assert prod in (0, 8, 16, 32) and prod_ms > 0 and after == res
    A.close()
