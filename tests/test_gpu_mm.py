"""The matrix-instruction products (product choice 32, and the residual of an unpinned refined
solve) at the edges of their tiles: clusters of 1 to 64 unknowns (tiles of 8 and 16 outputs,
K chunks of 16), ranks 1 to 32, right-hand sides around the tiles of 16 and the groups of 32
and 64, block scales far from 1, single zero and non-finite right-hand sides; against the same
blocks in numpy complex128.

Bounds: the FP32 product is held to 1e-5 per right-hand side as every product choice is (two
FP16 halves of 22 bits, FP32 sums: a few 1e-7); a refined solve of this well-conditioned
operator ends in complex64, a few 1e-7, held to 1e-5.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 7, 8, 9, 15, 16, 17, 31, 33, 48, 63, 64]


class Blocks:
    def __init__(self, seed, scale):
        rng = self.rng = np.random.default_rng(seed)
        self.off = np.concatenate([[0], np.cumsum(SIZES)])
        self.n = int(self.off[-1])
        self.perm = rng.permutation(self.n)
        n = len(SIZES)
        self.D = [scale * (4 * np.eye(m) + self.rand(m, m) / np.sqrt(2 * m)) for m in SIZES]
        self.near, self.far = [], []
        for i in range(n):
            for j in range(i + 1, n):
                m, w, kind = SIZES[i], SIZES[j], rng.integers(3)
                r, c = int(self.off[i]), int(self.off[j])
                if kind == 0:
                    self.near.append((r, c, scale * 0.1 * self.rand(m, w) / np.sqrt(m + w)))
                else:
                    k = int(rng.integers(1, min(m, w, 32) + 1))
                    # factors of very different size, rows of a factor too
                    g = 2.0 ** rng.integers(-20, 21)
                    U = g * self.rand(m, k) * 2.0 ** -np.arange(k)
                    V = scale * 0.1 / g * self.rand(k, w) / np.sqrt(m + w)
                    self.far.append((1, r, c, U, V))

    def rand(self, *s):
        return self.rng.normal(size=s) + 1j * self.rng.normal(size=s)

    def off_diag(self, v):
        z = np.zeros_like(v)
        for b in self.near + [(r, c, U @ V) for _, r, c, U, V in self.far]:
            r, c, B = b
            z[r:r + B.shape[0]] += B @ v[c:c + B.shape[1]]
            z[c:c + B.shape[1]] += B.T @ v[r:r + B.shape[0]]
        return z

    def diag(self, v, inv):
        return np.concatenate([(np.linalg.solve(d, v[a:b]) if inv else d @ v[a:b])
                               for d, a, b in zip(self.D, self.off, self.off[1:])])

    def series(self, r):
        y = x = self.diag(r, True)
        for _ in range(2):
            x = y - self.diag(self.off_diag(x), True)
        return x

    def operator(self):
        from paper_2307_03968_gb300.hm import HMatrix
        A = HMatrix.from_blocks(self.perm, self.off, self.D, self.near, self.far)
        A.factor_leaf()
        return A

    def vectors(self, nrhs):
        v = np.ascontiguousarray(self.rand(self.n, nrhs).T).astype(np.complex64)
        return v, v.astype(np.complex128).T[self.perm]

    def back(self, t):
        out = np.empty_like(t)
        out[self.perm] = t
        return out.T


def off_by(got, want):
    return (np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)).max()


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("nrhs", [4, 5, 15, 16, 17, 32, 33, 48, 64, 65, 130])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60, 2.0 ** -60])
def test_product_and_refined_solve(torch_cuda, nrhs, scale):
    B = Blocks(nrhs, scale)
    A = B.operator()
    x, xt = B.vectors(nrhs)
    x[1] = 0                                           # a zero right-hand side
    xt[:, 1] = 0
    xd = torch_cuda.from_numpy(x).cuda()
    yd = torch_cuda.empty_like(xd)
    A.set_tuning(nrhs, 32, 0)
    A.apply(xd, yd, n_levels=1, fp64_accumulate=False)
    want = B.back(B.diag(xt, False) + B.off_diag(xt))
    got = yd.cpu().numpy()
    keep = np.arange(nrhs) != 1
    assert np.all(got[1] == 0)
    assert off_by(got[keep], want[keep]) < 1e-5
    A.close()
    A = B.operator()                                   # not pinned: the solve's own choice
    b, bt = B.vectors(nrhs)
    bd = torch_cuda.from_numpy(b).cuda()
    s = B.series(bt)
    s = s + B.series(bt - B.diag(s, False) - B.off_diag(s))
    for _ in range(2):
        A.solve(bd, yd, n_terms=2, n_levels=1, refine=True)
        A.sync_status()
        assert off_by(yd.cpu().numpy(), B.back(s)) < 1e-5
    A.close()


def test_non_finite_right_hand_side_stays_alone(torch_cuda):
    from paper_2307_03968_gb300.hm import HmError, HM_ERR_DIVERGED
    B = Blocks(3, 1.0)
    A = B.operator()
    nrhs = 20
    x, xt = B.vectors(nrhs)
    x[7, 5] = np.inf
    x[18, 300] = np.nan
    xd = torch_cuda.from_numpy(x).cuda()
    yd = torch_cuda.empty_like(xd)
    A.set_tuning(nrhs, 32, 0)
    A.apply(xd, yd, n_levels=1, fp64_accumulate=False)
    got = yd.cpu().numpy()
    keep = [r for r in range(nrhs) if r not in (7, 18)]
    want = B.back(B.diag(xt, False) + B.off_diag(xt))
    assert off_by(got[keep], want[keep]) < 1e-5
    assert not np.isfinite(got[7]).all() and not np.isfinite(got[18]).all()
    A.close()
    A = B.operator()
    A.solve(xd, yd, n_terms=2, n_levels=1, refine=True)
    with pytest.raises(HmError) as e:
        A.sync_status()
    assert e.value.status == HM_ERR_DIVERGED
    # nothing of it stays behind for the next call
    b, bt = B.vectors(nrhs)
    bd = torch_cuda.from_numpy(b).cuda()
    A.solve(bd, yd, n_terms=2, n_levels=1, refine=True)
    A.sync_status()
    s = B.series(bt)
    s = s + B.series(bt - B.diag(s, False) - B.off_diag(s))
    assert off_by(yd.cpu().numpy(), B.back(s)) < 1e-5
    A.close()
