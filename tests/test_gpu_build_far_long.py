"""Far blocks of hm_build that the re-compression gives a CTA each (rank above 16 and a side above 256)
against the oracle's dense blocks, beside the form that test_gpu_build_far.py checks.

tol = 1e-5: the two truncations (ACA, re-compression) leave 2e-5 of the block (Frobenius).  Its
entries are FP32 evaluations, 2e-5 off at most (as the near blocks are held to), and so are the row and
the column of each of the k crosses that the block is made of: 2e-5 (1 + sqrt(k)) if they are
independent, 1.6e-4 in all at rank 36 (measured: 6e-5; the noise makes the rank, the block itself is of
rank 12 to 1e-5).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_long_blocks_of_high_rank_match_oracle():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import plate
    from oracle.rwg import RWGMesh
    from paper_2307_03968_gb300.hm import HMatrix
    xyz, tri = plate((6.0, 0.4), (120, 8))
    mesh = RWGMesh(xyz, tri)
    A = HMatrix.build(xyz, tri, leaf_size=40, arity=2, adm=1.0, aca_tol=1e-5, levels=-1)
    P = A.perm()
    seen = 0
    for lev in range(1, A.info().n_levels + 1):
        r0, c0, m, w, k = A.blocks(lev)
        for idx in np.nonzero((k > 16) & (np.maximum(m, w) > 256))[0][:6]:
            U, V = A.block(lev, idx)
            Z = mesh.fill(P[r0[idx]:r0[idx] + m[idx]], P[c0[idx]:c0[idx] + w[idx]])
            assert np.linalg.norm(U @ V - Z) <= (2e-5 + 2e-5 * (1 + np.sqrt(k[idx]))) * np.linalg.norm(Z), (lev, idx, k[idx])
            seen += 1
    A.close()
    assert seen >= 2
