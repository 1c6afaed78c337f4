"""A server whose HBM budget holds its operators keeps them, whatever the many-right-hand-side kernels
pack beside them: three operators that fit the budget, whose operand streams do not, are each built
once and never evicted, and the streams stay within the budget.  Results as of the same requests
solved alone (1e-5, as in the other server tests)."""

import numpy as np
import pytest

from hm_testutil import rel_err

pytestmark = pytest.mark.gpu


def test_operand_streams_evict_no_operator():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import icosphere
    from paper_2307_03968_gb300.hm import HMatrix, Server
    nrhs = 32
    opts = dict(leaf_size=64, arity=8, adm=2.0, aca_tol=1e-4)
    sopts = dict(n_terms=2, n_levels=1, refine=True)
    meshes = [icosphere(4, 0.7 + 0.1 * i) for i in range(3)]   # 7,680 unknowns each
    rng = np.random.default_rng(3)
    base, packed, want, rhs = [], [], [], []
    for xyz, tri in meshes:
        A = HMatrix.build(xyz, tri, levels=1, **opts)
        A.factor_leaf()
        b = (rng.normal(size=(nrhs, A.n)) + 1j * rng.normal(size=(nrhs, A.n))).astype(np.complex64)
        bt = torch.from_numpy(b).cuda()
        xt = torch.empty_like(bt)
        A.set_tuning(nrhs, 16, 1017)                           # without operand streams
        A.solve(bt, xt, **sopts)
        torch.cuda.synchronize()
        base.append(A.info().device_bytes)
        want.append(xt.cpu().numpy())
        A.set_tuning(nrhs, 32, 1018)
        A.solve(bt, xt, **sopts)
        torch.cuda.synchronize()
        packed.append(A.info().device_bytes)
        rhs.append(b)
        A.close()
    estimate = 60 * 1024 * max(b.shape[1] for b in rhs)        # an operator's size before its first build
    budget = int(max(1.1 * sum(base), sum(base) - min(base) + 1.02 * estimate))
    assert budget < 0.8 * sum(packed)
    srv = Server(n_slots=3, hbm_budget_bytes=budget, max_batch_rhs=nrhs)
    ops = [srv.add_mesh(xyz, tri, levels=1, **opts, **sopts)[0] for xyz, tri in meshes]
    for _ in range(3):
        for k in (0, 1, 2, 1, 0, 2):
            x, _ = srv.wait(srv.submit(ops[k], rhs[k]))
            assert rel_err(x, want[k]) < 1e-5
    info = srv.info()
    assert info.builds == 3 and info.evictions == 0
    assert info.peak_resident_bytes <= 1.02 * budget
    srv.close()
