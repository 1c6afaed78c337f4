"""An infinite or NaN entry of a right-hand side reaches the outputs that its blocks couple it to and no
others, in the matrix-instruction product (32) and residual (1018) as in the FP32 kernels: nothing of
it gets into the scales of the other entries, which are far from 1 here.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, complex(0, np.inf)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 40, 2.0 ** -40])
def test_reaches_only_its_neighbours(bad, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(2)
    m, leaves, nrhs = 30, 12, 20
    n = m * leaves

    def rand(*s):
        return (rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64).astype(np.complex128)

    D = [rand(m, m) + 8 * np.eye(m) for _ in range(leaves)]
    near = [(m * i, m * (i + 1), rand(m, m)) for i in range(0, leaves - 1, 2)]
    far = [(1, m * i, m * (i + 3), rand(m, 5), rand(5, m)) for i in range(0, leaves - 3, 4)]
    M = np.zeros((n, n), np.complex128)
    for i, d in enumerate(D):
        M[m * i:m * i + m, m * i:m * i + m] = d
    for r, c, B in near + [(r, c, U @ V) for _, r, c, U, V in far]:
        M[r:r + m, c:c + m] = B
        M[c:c + m, r:r + m] = B.T
    A = HMatrix.from_blocks(np.arange(n), m * np.arange(leaves + 1), D, near, far)
    A.factor_leaf()
    x = (scale * rand(nrhs, n)).astype(np.complex64)
    at = 4 * m + 7                                         # coupled to leaves 4 (itself), 5 (near) and 7 (far)
    x[3, at] = bad
    reach = np.zeros((nrhs, n), bool)
    reach[3] = np.repeat(np.isin(np.arange(leaves), (4, 5, 7)), m)
    clean = np.where(np.isfinite(x), x, 0).astype(np.complex128)
    want = clean @ M.T
    xt = torch.tensor(x, device="cuda")
    yt = torch.empty_like(xt)
    A.set_tuning(nrhs, 32, 1018)
    A.apply(xt, yt, n_levels=1, fp64_accumulate=False)
    y = yt.cpu().numpy()
    A.residual(torch.zeros_like(xt), xt, yt, n_levels=1)
    for got, ref in ((y, want), (yt.cpu().numpy(), -want)):
        assert not np.isfinite(got[reach]).any()
        assert np.abs(got - ref)[~reach].max() < 1e-5 * np.abs(ref).max()
    A.close()
