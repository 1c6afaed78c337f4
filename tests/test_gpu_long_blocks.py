"""Low-rank blocks longer than 64: rank panels of the product, CTA-wide residual products, and
all the levels' residual products in one launch (more levels than one launch takes), against
numpy on the same blocks.

Ragged leaves, blocks between unions of them, ranks around the panel (8), the four rank rows of
a warp and the pass (32).  Single-precision sums of at most 1,024 terms leave a few 1e-7 of
|A| |x|, held to 5e-6; FP64-class results are rounded to single once (6e-8), held to 2e-7.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [65, 30, 64, 1, 129, 40, 33, 500, 7, 66]
RANKS = [1, 3, 7, 8, 9, 16, 31, 32, 33, 70]


@pytest.mark.parametrize("levels,nrhs", [(a, b) for a in (1, 3, 10) for b in (1, 2, 5, 17)] + [(0, 1), (0, 2)])
def test_long_blocks_match_numpy(levels, nrhs):
    """levels = 0: so many blocks of 66 on one level that each is a warp's."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(100 * levels + nrhs)
    sizes = SIZES if levels else [66] * 90
    off = np.concatenate([[0], np.cumsum(sizes)])
    n, nl = int(off[-1]), len(sizes)

    def rand(*s):
        return (rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64).astype(np.complex128)

    D = [np.eye(m) + 0.3 * rand(m, m) / np.sqrt(2 * m) for m in sizes]
    D = [d.astype(np.complex64).astype(np.complex128) for d in D]
    near = [(int(off[0]), int(off[4]), rand(sizes[0], sizes[4]))]
    far = []
    for lev in range(1, levels + 1):
        for q in range(4):
            w = min(lev, nl // 2)                          # leaves of a cluster
            i = int(rng.integers(0, nl - 2 * w + 1))
            j = int(rng.integers(i + w, nl - w + 1))
            m, c, k = off[i + w] - off[i], off[j + w] - off[j], RANKS[(3 * lev + q) % len(RANKS)]
            far.append((lev, int(off[i]), int(off[j]), rand(m, k) / k, rand(k, c)))
    if not levels:
        far = [(1, int(off[i]), int(off[j]), rand(66, 2), rand(2, 66)) for i in range(nl) for j in range(i + 1, nl)
               if (i, j) != (0, 4)]
    far = [(a, b, c, U.astype(np.complex64).astype(np.complex128), V) for a, b, c, U, V in far]
    A = HMatrix.from_blocks(np.arange(n), off, D, near, far)
    A.factor_leaf()
    M = np.zeros((n, n), np.complex128)
    for i, d in enumerate(D):
        M[off[i]:off[i + 1], off[i]:off[i + 1]] = d
    for r, c, B in near + [(r, c, U @ V) for _, r, c, U, V in far]:
        M[r:r + B.shape[0], c:c + B.shape[1]] += B
        M[c:c + B.shape[1], r:r + B.shape[0]] += B.T
    x, b = (rand(nrhs, n).astype(np.complex64) for _ in range(2))
    ref = x.astype(np.complex128) @ M.T
    scale = np.abs(x) @ np.abs(M).T
    for k in range(len(far)):                              # |U| |V| |x| bounds the two-stage sums
        _, r, c, U, V = far[k]
        scale[:, r:r + len(U)] += np.abs(x[:, c:c + V.shape[1]]) @ (np.abs(U) @ np.abs(V)).T
        scale[:, c:c + V.shape[1]] += np.abs(x[:, r:r + len(U)]) @ (np.abs(U) @ np.abs(V))
    xt, y = torch.tensor(x, device="cuda"), torch.empty(nrhs, n, dtype=torch.complex64, device="cuda")
    A.apply(xt, y, n_levels=-1, fp64_accumulate=False)
    assert np.max(np.abs(y.cpu().numpy() - ref) / scale) < 5e-6
    A.apply(xt, y, n_levels=-1, fp64_accumulate=True)
    assert np.max(np.abs(y.cpu().numpy() - ref) / np.maximum(np.abs(ref), 1e-6 * scale)) < 2e-7
    y0 = y.clone()
    A.apply(xt, y, n_levels=-1, fp64_accumulate=True)
    assert torch.equal(y, y0)                              # a fixed order of the sums
    r = torch.empty_like(y)
    A.residual(torch.tensor(b, device="cuda"), xt, r, n_levels=-1)
    want = b - ref
    assert np.max(np.abs(r.cpu().numpy() - want) / np.maximum(np.abs(want), 1e-6 * scale)) < 2e-7
