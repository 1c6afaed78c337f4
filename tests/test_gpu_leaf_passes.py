"""The leaf passes (x = y - D^{-1} z and the passes fused with it) where their grids change:
row chunks of 64 for few long leaves, four right-hand sides a CTA for many leaves, ragged
counts of both, against the same series in numpy on the same blocks.

Random blocks with D diagonally dominant (condition about 3) and one dense coupling block
of norm about 0.1: complex64 storage and sums leave a few 1e-7, held to 1e-5.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = {
    "long_few": [300, 65, 64, 1],
    "chunk_edges": [128, 129, 63],
    "one_leaf": [1050],
    "many_short": [7] * 700,
    "many_64": [64] * 310,
    "many_65": [65] * 310,
}


@pytest.mark.parametrize("name,nrhs", [("long_few", 1), ("long_few", 3), ("chunk_edges", 2), ("one_leaf", 1),
                                       ("many_short", 5), ("many_64", 9), ("many_65", 8), ("many_64", 3)])
@pytest.mark.parametrize("refine", [False, True])
def test_leaf_passes_match_numpy(name, nrhs, refine):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    sizes = SHAPES[name]
    rng = np.random.default_rng(len(sizes) * 100 + nrhs)
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = off[-1]
    perm = rng.permutation(n)

    def rand(*s):
        return rng.normal(size=s) + 1j * rng.normal(size=s)

    D = [np.eye(m) + 0.3 * rand(m, m) / np.sqrt(2 * m) for m in sizes]
    near = []
    if len(sizes) > 1:
        near = [(0, int(off[1]), 0.1 * rand(sizes[0], sizes[1]) / np.sqrt(2 * max(sizes[:2])))]
    A = HMatrix.from_blocks(perm, off, D, near, [])
    A.factor_leaf()
    b = rand(nrhs, n).astype(np.complex64)

    def inv(v):
        return np.concatenate([np.linalg.solve(D[i], v[off[i]:off[i + 1]]) for i in range(len(sizes))])

    def off_diag(v):
        z = np.zeros_like(v)
        for r, c, B in near:
            z[r:r + B.shape[0]] += B @ v[c:c + B.shape[1]]
            z[c:c + B.shape[1]] += B.T @ v[r:r + B.shape[0]]
        return z

    def series(r):
        y = x = inv(r)
        for _ in range(2):
            x = y - inv(off_diag(x))
        return x

    bt = b.astype(np.complex128).T[perm]
    ref = series(bt)
    if refine:
        Dx = np.concatenate([D[i] @ ref[off[i]:off[i + 1]] for i in range(len(sizes))])
        ref = ref + series(bt - Dx - off_diag(ref))
    want = np.empty_like(ref)
    want[perm] = ref
    bd = torch.from_numpy(b).cuda()
    x = torch.empty_like(bd)
    for _ in range(2):                      # the second pass finds the vectors the first one left
        A.solve(bd, x, n_terms=2, n_levels=1, refine=refine, graph=False)
        A.sync_status()
        got = x.cpu().numpy().T
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    A.close()
