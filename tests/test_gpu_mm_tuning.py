"""hm_get_tuning names the residual kernel that refined solves run, and hm_set_tuning takes what it
named: the pinned solve enqueues the same kernels, and hm_residual runs it too (a fixed order of
the sums: equal bit for bit over two calls).
"""

import pytest

from test_gpu_mm import Blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [20, 70])
def test_reported_choice_can_be_pinned(nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B = Blocks(nrhs, 1.0)
    A, P = B.operator(), B.operator()
    b, _ = B.vectors(nrhs)
    bt = torch.from_numpy(b).cuda()
    xt, r = torch.empty_like(bt), torch.empty_like(bt)
    free = A.solve(bt, xt, n_terms=2, n_levels=1, refine=True, info=True)
    prod, res, _, _ = A.tuning(nrhs)
    assert res == 1018                                     # above 16 right-hand sides always
    P.set_tuning(nrhs, prod, res)
    pinned = P.solve(bt, xt, n_terms=2, n_levels=1, refine=True, info=True)
    assert pinned.kernel_launches == free.kernel_launches
    assert P.tuning(nrhs)[:2] == (prod, res)
    P.residual(bt, xt, r, n_levels=1)
    again = torch.empty_like(r)
    P.residual(bt, xt, again, n_levels=1)
    assert torch.equal(r, again)
    P.set_tuning(nrhs, prod, 0)
    P.residual(bt, xt, again, n_levels=1)
    assert (r - again).abs().max() <= 1e-5 * bt.abs().max()
    for M in (A, P):
        M.close()
