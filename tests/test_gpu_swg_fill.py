"""Near blocks of the V-EFIE fill over the chunk sizes it works in (32 x 32 faces): leaves
of a few faces, at 32, 33 and above, homogeneous cells (eps_r = 1: no contrast) among the
others; every entry of every near block against the oracle's complex128 fill, relative to the
block's largest entry, <= 2e-5 as for the other near blocks (FP32 quadrature).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf", [((2, 2, 2), 7), ((2, 2, 2), 32), ((3, 2, 2), 33), ((3, 3, 2), 70), ((1, 1, 1), 9)])
def test_near_blocks_match_oracle(n, leaf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import box_tets, random_permittivity
    from oracle.swg import SWGMesh
    from paper_2307_03968_gb300.hm import HMatrix
    xyz, tet = box_tets(tuple(0.07 * k for k in n), n)
    eps = random_permittivity(len(tet), 2.0, 6.0, seed=sum(n))
    eps[::5] = 1.0
    mesh = SWGMesh(xyz, tet, eps)
    A = HMatrix.build(xyz, tet, eps_r=eps, leaf_size=leaf, arity=2, adm=1.0, aca_tol=1e-4, levels=-1)
    P = A.perm()
    r0, c0, m, w, k = A.blocks(1)
    seen = 0
    for idx in np.nonzero(k == 0)[0]:
        ref = mesh.fill(P[r0[idx]:r0[idx] + m[idx]], P[c0[idx]:c0[idx] + w[idx]])
        B = A.block(1, idx)
        assert np.abs(B - ref).max() <= 2e-5 * np.abs(ref).max(), idx
        seen += 1
    A.close()
    assert seen > 0
