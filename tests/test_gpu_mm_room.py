"""The matrix-instruction kernels' operand streams are an addition to an operator that works without
them: they take at most half of the memory that is free, so that a call on an operator does not
take the rest of the device from others.  Without them the calls run the other kernels, with the same
results (1e-5 of each other: FP32 sums in another order), and keep to them; a pinned choice asks again.
"""

import gc

import pytest

from test_gpu_mm_accuracy import Operator

pytestmark = pytest.mark.gpu


# left: what is free when the product is tuned, in tenths of the streams (at their unpadded size): too
# little for them, and enough for them but not for the operand tiles with them
@pytest.mark.parametrize("left", [19, 28])
def test_streams_leave_room(left):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = Operator(1.0)
    A, T = P.handle(), P.handle()
    nrhs = 40
    xt = torch.tensor(P.vectors("even", nrhs), device="cuda")
    y, ref, x, xref = (torch.empty_like(xt) for _ in range(4))
    T.apply(xt, ref, n_levels=1, fp64_accumulate=False)    # with room
    T.solve(xt, xref, n_terms=1, n_levels=1, refine=True, graph=False)
    assert T.tuning(nrhs)[1] == 1018
    streams = 2 * 8 * (A.info().near_elems + sum(A.info().far_elems))
    vectors = 16 * 8 * 64 * (P.n + 64)                     # the product's work vectors at the bucket's 64 right-hand sides
    gc.collect()                                           # nothing of earlier tests is given back in between
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held, free = A.info().device_bytes, torch.cuda.mem_get_info()[0]
    more = torch.empty(512 << 20, dtype=torch.uint8, device="cuda")
    fill = torch.empty(free - more.numel() - vectors - left * streams // 10, dtype=torch.uint8, device="cuda")
    taken = after = 0
    try:
        A.apply(xt, y, n_levels=1, fp64_accumulate=False)
        torch.cuda.synchronize()
        taken, after = A.info().device_bytes - held, torch.cuda.mem_get_info()[0]
        del more
        torch.cuda.empty_cache()
        A.solve(xt, x, n_terms=1, n_levels=1, refine=True, graph=False)
        A.sync_status()
        choice = A.tuning(nrhs)[:2]
    finally:
        del fill
        torch.cuda.empty_cache()
    assert taken < vectors + streams // 2 and after > streams
    assert choice == (16, 1017)
    for got, want in ((y, ref), (x, xref)):
        assert ((got - want).norm(dim=1) / want.norm(dim=1)).max() < 1e-5
    A.set_tuning(nrhs, 32, 1018)
    A.apply(xt, y, n_levels=1, fp64_accumulate=False)
    assert ((y - ref).norm(dim=1) / ref.norm(dim=1)).max() < 1e-5
    assert A.info().device_bytes - held - taken >= streams
    A.close()
    T.close()
