"""Far blocks of hm_build over the ranks and block lengths at which the ACA and the
re-compression change their thread groups: ranks up to 8, 16 and above (one warp per
block, or a CTA), blocks shorter and longer than 256, rows of up to 32 and above.

Each checked block:
- is in the form the re-compression gives it, a singular value decomposition: the rows
  of V orthonormal, the columns of U orthogonal with non-increasing norms.  The factors
  are FP32 rows formed from FP64 rotations of rows orthonormal to FP32 (Gram-Schmidt
  twice), so inner products are held to 1e-5 (a few FP32 roundings, 6e-8 each, over up
  to 48 rows);
- for tolerances well above the noise of FP32 entries (1e-4 and more), U V is within
  5 x tol (relative, Frobenius) of the oracle's dense block, as for the other far blocks:
  two truncations at tol, one each in ACA and re-compression.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size,n,leaf,tol,want", [
    ((0.6, 0.6), (12, 12), 16, 1e-2, dict(max_rank=8)),                       # short rows, ranks of one warp's 8
    ((1.0, 1.0), (20, 20), 31, 1e-4, dict(max_rank=16)),                      # odd leaves, ranks up to 16
    ((6.0, 0.4), (120, 8), 40, 1e-5, dict(min_rank=17, min_side=257)),        # long blocks of high rank: a CTA each
])
def test_far_blocks_by_rank_and_length(size, n, leaf, tol, want):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import plate
    from oracle.rwg import RWGMesh
    from paper_2307_03968_gb300.hm import HMatrix
    xyz, tri = plate(size, n)
    mesh = RWGMesh(xyz, tri)
    A = HMatrix.build(xyz, tri, leaf_size=leaf, arity=2, adm=1.0, aca_tol=tol, levels=-1)
    P = A.perm()
    ranks, sides = [], []
    for lev in range(1, A.info().n_levels + 1):
        r0, c0, m, w, k = A.blocks(lev)
        far = np.nonzero(k > 0)[0]
        for idx in far[::max(1, len(far) // 12)]:
            U, V = A.block(lev, idx)
            if k[idx] > 1:
                assert np.abs(V @ V.conj().T - np.eye(k[idx])).max() < 1e-5, (lev, idx, k[idx])
                s = np.linalg.norm(U, axis=0)
                gram = U.conj().T @ U
                assert np.abs(gram - np.diag(np.diag(gram))).max() < 1e-5 * s[0] ** 2, (lev, idx, k[idx])
                assert np.all(s[1:] <= s[:-1] * (1 + 1e-5))
            if tol >= 1e-4:
                Z = mesh.fill(P[r0[idx]:r0[idx] + m[idx]], P[c0[idx]:c0[idx] + w[idx]])
                assert np.linalg.norm(U @ V - Z) <= 5 * tol * np.linalg.norm(Z), (lev, idx, k[idx])
            ranks.append(k[idx])
            sides.append(max(m[idx], w[idx]))
    A.close()
    assert len(ranks) >= 10
    assert min(ranks) <= want.get("max_rank", 48) and max(ranks) >= want.get("min_rank", 1)
    assert max(sides) >= want.get("min_side", 1)
