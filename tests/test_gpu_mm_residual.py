"""The FP64-class residual on the matrix instructions (residual choice 1018, the one that unpinned
refined solves run) by itself, against that of the owner-computes kernel on the FP32 pipes (1017).

b = fl32(A x), so that the true residual is about 2^-25 of |A x| and what the sums err by shows.
Errors are per output, beyond the rounding of the output, in units of the sum of the moduli of
its terms (through a low-rank block's two factors): right-hand sides of even size, an
excitation of one leaf with everything else at 2^-30 of it, entries spread over 2^-30.  Digits reach
48 bits below the largest entry of a chunk of 16 K (of a row of the block, and of a right-hand
side), products below 2^-45 of both are left out: with 32 products a chunk and part all at their
largest 2^-39 of that scale, held to 2^-34 of the sum of the moduli (which is seldom less than the
scale over 30, 2^-5), as the FP64-class kernels are elsewhere to 2^-30; the rms to 1.25 of that of 1017.
"""

import numpy as np
import pytest

from test_gpu_mm_accuracy import Operator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def operator():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = Operator(1.0)
    A = P.handle()
    yield P, A
    A.close()


def residual(A, b, x, choice):
    import torch
    xt, bt = torch.tensor(x, device="cuda"), torch.tensor(b, device="cuda")
    r = torch.full_like(xt, float("nan"))
    A.set_tuning(len(x), 0, choice)
    A.residual(bt, xt, r, n_levels=1)
    return r.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("kind", ["even", "one leaf", "spread"])
@pytest.mark.parametrize("nrhs", [4, 16, 17, 40])
def test_as_accurate_as_the_owner_kernel(operator, kind, nrhs):
    P, A = operator
    x = P.vectors(kind, nrhs)
    ax = x.astype(np.complex128) @ P.M.T
    b = ax.astype(np.complex64)
    want = b - ax
    scale = np.abs(x) @ (P.A[0] + P.A[1]).T
    err = {}
    for choice in (1017, 1018):
        e = np.abs(residual(A, b, x, choice) - want)
        err[choice] = np.maximum(e - 2.0 ** -23 * np.abs(want), 0) / scale
    rms = {c: np.sqrt(np.mean(e ** 2)) for c, e in err.items()}
    print("log2 of the error: 1017 rms %.1f max %.1f; 1018 rms %.1f max %.1f" %
          tuple(np.log2(v) for c in (1017, 1018) for v in (rms[c], err[c].max())))
    assert err[1018].max() < 2.0 ** -34
    assert rms[1018] <= 1.25 * rms[1017]


def test_exact_answers(operator):
    """x = 0 gives b bit for bit; a scaled unit vector gives a column of the operator (2^-23 of its own
    rounding, 2^-34 of the terms' moduli, which the scales keep above the smallest float)."""
    P, A = operator
    nrhs = 20
    rng = np.random.default_rng(1)
    b = (rng.normal(size=(nrhs, P.n)) + 1j * rng.normal(size=(nrhs, P.n))).astype(np.complex64)
    x = np.zeros_like(b)
    assert np.array_equal(residual(A, b, x, 1018), b)
    x[np.arange(nrhs), rng.choice(P.n, nrhs, replace=False)] = \
        ((rng.normal(size=nrhs) + 1j * rng.normal(size=nrhs)) * 2.0 ** (10 * (np.arange(nrhs) - 10))).astype(np.complex64)
    want = -(x.astype(np.complex128) @ P.M.T)
    scale = np.abs(x) @ (P.A[0] + P.A[1]).T
    got = residual(A, np.zeros_like(b), x, 1018)
    on = scale > 0
    assert np.all(got[~on] == 0)
    assert np.all(np.abs(got - want)[on] <= 2.0 ** -23 * np.abs(want)[on] + 2.0 ** -34 * scale[on])


@pytest.mark.parametrize("value", [1 - 2.0 ** -24, 1 - 2.0 ** -10 - 2.0 ** -19 + 2.0 ** -24])
def test_largest_digits_of_one_sign(value):
    """All entries of block and vector the same, digits near their largest and of one sign: the sums
    of the digit products are then as large as they can be.  Every term is exactly value^2."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_03968_gb300.hm import HMatrix
    v = np.float64(np.float32(value))
    m = 64
    B = np.full((m, m), v * (1 + 1j))
    A = HMatrix.from_blocks(np.arange(2 * m), np.array([0, m, 2 * m]), [np.eye(m) + 0j] * 2, [(0, m, B)], [])
    A.factor_leaf()
    x = np.full((20, 2 * m), v * (1 - 1j)).astype(np.complex64)
    ax = x.astype(np.complex128).copy()
    ax[:, :m] += x[:, m:].astype(np.complex128) @ B.T
    ax[:, m:] += x[:, :m].astype(np.complex128) @ B
    b = ax.astype(np.complex64)
    want = b - ax
    got = residual(A, b, x, 1018)
    A.close()
    assert np.abs(got - want).max() <= 2.0 ** -23 * np.abs(want).max() + 2.0 ** -43 * 2 * m * v * v
