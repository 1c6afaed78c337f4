"""The matrix-instruction products (product choice 32) at the ends of the FP32 range: factors of
a low-rank block of very different size, blocks and vectors near the largest and the smallest
floats.  Every product and every term of it is a normal FP32 number, so the FP32 kernels (choice
16) are exact to their rounding here; both are held to 1e-5 of numpy complex128 per right-hand
side, as every product choice is, over the rows that only the block reaches.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("u,v,x,rank", [
    (-118, 16, 0, 5), (-112, 7, 0, 5), (16, -118, 0, 3), (-60, -60, 60, 8),     # U, V, x: powers of two
    (-10, -10, 124, 4), (-30, -30, 125, 4), (50, 60, -30, 4), (-20, 0, -98, 4),
    (124, None, -20, 0), (-120, None, 60, 0), (-10, None, 125, 0),               # a dense block
])
@pytest.mark.parametrize("zero_row", [False, True])
def test_extreme_scales(u, v, x, rank, zero_row):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(rank)
    sizes, nrhs = [17, 30], 6
    off = np.array([0, 17, 47])

    def rand(e, *s):                                       # components within [1/2, 1] 2^e
        a = rng.uniform(0.5, 1.0, size=s) + 1j * rng.uniform(0.5, 1.0, size=s)
        return (a * 2.0 ** e).astype(np.complex64).astype(np.complex128)

    D = [np.eye(m) + 0j for m in sizes]
    if rank:
        U, V = rand(u, sizes[0], rank), rand(v, rank, sizes[1])
        if zero_row:                                       # gives nothing, whatever its partner holds
            V[0] = 0
            U[:, 0] = rand(u, sizes[0])
        A = HMatrix.from_blocks(np.arange(47), off, D, [], [(1, 0, 17, U, V)])
        B = U @ V
    else:
        B = rand(u, *sizes)
        A = HMatrix.from_blocks(np.arange(47), off, D, [(0, 17, B)], [])
    A.factor_leaf()
    for rows, cols, M in [(slice(0, 17), slice(17, 47), B), (slice(17, 47), slice(0, 17), B.T)]:
        xv = np.zeros((nrhs, 47), np.complex64)
        xv[:, cols] = rand(x, nrhs, xv[:, cols].shape[1])
        want = xv[:, cols].astype(np.complex128) @ M.T
        xt = torch.tensor(xv, device="cuda")
        yt = torch.empty_like(xt)
        for choice in (16, 32):
            A.set_tuning(nrhs, choice, 0)
            A.apply(xt, yt, n_levels=1, fp64_accumulate=False)
            got = yt.cpu().numpy()[:, rows].astype(np.complex128)
            err = np.linalg.norm((got - want) * 2.0 ** -100, axis=1) / np.linalg.norm(want * 2.0 ** -100, axis=1)
            assert err.max() < 1e-5, (choice, err.max())
    A.close()
