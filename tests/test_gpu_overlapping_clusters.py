"""A user's own blocks may couple, on one level, a leaf and a union of leaves that holds it: the
output rows of such clusters overlap.  The owner-computes residuals (pinned, and of unpinned
refined solves) store the sums of whole clusters, so they must leave such levels to the kernels
that add.  Against the same blocks in numpy complex128: the residual of FP64-class sums rounded to
single once, held to 2e-7 of the sum of the moduli; the refined solve of this well-conditioned
operator to 1e-5 (complex64, a few 1e-7).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [5, 20, 40])
def test_leaf_inside_a_union_on_one_level(nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(nrhs)
    sizes = [int(v) for v in rng.integers(5, 17, 24)]
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])

    def rand(*s):
        return (rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64).astype(np.complex128)

    D = [(4 * np.eye(m) + rand(m, m) / 8).astype(np.complex64).astype(np.complex128) for m in sizes]
    far = []
    for i in range(0, 24, 2):                              # spans of one to three leaves, starting inside one another
        for j in range(i + 4, 22, 3):
            for a, b, c, d in [(i, i + 2, j, j + 1), (i + 1, i + 2, j, j + 2), (i + 1, i + 3, j, j + 2)]:
                m, w = int(off[b] - off[a]), int(off[d] - off[c])
                k = int(rng.integers(1, 6))
                far.append((1, int(off[a]), int(off[c]), 0.02 * rand(m, k), 0.1 * rand(k, w)))
    far = [(lev, r, c, U.astype(np.complex64).astype(np.complex128), V.astype(np.complex64).astype(np.complex128))
           for lev, r, c, U, V in far]
    Minv, M, S = (np.zeros((n, n), np.complex128) for _ in range(3))
    for i, d in enumerate(D):
        s = slice(off[i], off[i + 1])
        M[s, s], Minv[s, s], S[s, s] = d, np.linalg.inv(d), np.abs(d)
    F = np.zeros((n, n), np.complex128)
    for _, r, c, U, V in far:
        h, w = U.shape[0], V.shape[1]
        F[r:r + h, c:c + w] += U @ V
        F[c:c + w, r:r + h] += (U @ V).T
        S[r:r + h, c:c + w] += np.abs(U) @ np.abs(V)
        S[c:c + w, r:r + h] += (np.abs(U) @ np.abs(V)).T
    M += F
    A = HMatrix.from_blocks(np.arange(n), off, D, [], far)
    A.factor_leaf()
    x, b = (rand(nrhs, n).astype(np.complex64) for _ in range(2))
    xt, bt = torch.tensor(x, device="cuda"), torch.tensor(b, device="cuda")
    out = torch.empty_like(xt)

    def series(r):
        y = v = r @ Minv.T
        for _ in range(2):
            v = y - (v @ F.T) @ Minv.T
        return v

    want = series(b.astype(np.complex128))
    want = want + series(b - want @ M.T)
    A.solve(bt, out, n_terms=2, n_levels=1, refine=True)
    A.sync_status()
    got = out.cpu().numpy()
    assert (np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)).max() < 1e-5
    scale = np.abs(b) + np.abs(x) @ S.real.T
    for res in (None, 1017):
        if res is not None:
            A.set_tuning(nrhs, 0, res)
        A.residual(bt, xt, out, n_levels=1)
        assert np.max(np.abs(out.cpu().numpy() - (b - x.astype(np.complex128) @ M.T)) / scale) < 2e-7, res
    A.close()
