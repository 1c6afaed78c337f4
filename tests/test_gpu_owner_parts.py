"""The owner-computes residual with its clusters cut into parts, groups of 8 and 16 right-hand
sides, pairs at odd counts, and the gather over four right-hand sides, against numpy on the same
blocks.

Ragged leaves (one of them long, without blocks of its own), dense and low-rank blocks between
all other pairs: 19 to 45 products a cluster, cut into 2 to 5 parts.  FP64-class sums rounded to
single once (6e-8), held to 2e-7.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaves,nrhs", [(20, 5), (20, 17), (46, 8), (46, 33), (46, 130)])
def test_owner_parts_match_numpy(leaves, nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(leaves + nrhs)
    sizes = [int(v) for v in rng.integers(1, 65, leaves)] + [1100]
    sizes[3], sizes[5] = 64, 1
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])

    def rand(*s):
        return (rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64).astype(np.complex128)

    D = [rand(m, m) for m in sizes[:-1]] + [np.diag(rand(sizes[-1])) + 0j]
    near, far = [], []
    for i in range(leaves):
        for j in range(i + 1, leaves):
            if rng.random() < 0.3:
                near.append((int(off[i]), int(off[j]), rand(sizes[i], sizes[j])))
            else:
                k = int(rng.integers(1, 33))
                far.append((1, int(off[i]), int(off[j]), rand(sizes[i], k), rand(k, sizes[j])))
    A = HMatrix.from_blocks(np.arange(n), off, D, near, far)
    A.factor_leaf()
    M, S = np.zeros((n, n), np.complex128), np.zeros((n, n))
    for i, d in enumerate(D):
        M[off[i]:off[i + 1], off[i]:off[i + 1]] = d
    S[:] = np.abs(M)
    for r, c, B, bound in [(r, c, B, np.abs(B)) for r, c, B in near] + \
                          [(r, c, U @ V, np.abs(U) @ np.abs(V)) for _, r, c, U, V in far]:
        h, w = B.shape
        M[r:r + h, c:c + w] = B
        M[c:c + w, r:r + h] = B.T
        S[r:r + h, c:c + w] = bound
        S[c:c + w, r:r + h] = bound.T
    x, b = (rand(nrhs, n).astype(np.complex64) for _ in range(2))
    ax = x.astype(np.complex128) @ M.T
    want = b - ax
    scale = np.maximum(np.abs(want), 1e-6 * (np.abs(x) @ S.T))
    A.set_tuning(nrhs, 16, 1017)
    xt, bt = torch.tensor(x, device="cuda"), torch.tensor(b, device="cuda")
    r = torch.empty_like(xt)
    rn, bn = A.residual(bt, xt, r, n_levels=1)
    assert np.max(np.abs(r.cpu().numpy() - want) / scale) < 2e-7
    assert np.allclose(rn, np.sum(np.abs(want) ** 2, 1), rtol=1e-6)
    assert np.allclose(bn, np.sum(np.abs(b.astype(np.complex128)) ** 2, 1), rtol=1e-12)
    r2 = torch.empty_like(r)
    A.residual(bt, xt, r2, n_levels=1)
    assert torch.equal(r, r2)                              # a fixed order of the sums
