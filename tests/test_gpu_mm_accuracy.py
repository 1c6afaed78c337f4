"""Accuracy of the matrix-instruction product (choice 32) against that of the FP32 kernel it stands
beside (choice 16): it is chosen by time alone, so it may not be the less accurate one.

Errors are per output and per real part, in units of the sum of the moduli of the part's own
terms (for the real part sum |Re a Re x| + |Im a Im x|, through a low-rank block's two factors),
so that neither a large part nor a large cluster hides a small one: right-hand sides of even
size, an excitation of one leaf with everything else at 2^-30 of it, entries spread over 2^-30, and blocks with
imaginary parts of 2^-30 of the real ones (fine meshes have them), with real vectors.

Bounds: three parts of 8 bits hold an FP32 number exactly; the products left out are 2^-25 of a
term, the tensor core truncates the last two of twelve sums of a chunk of 16 K at the chunk's own
size (2 x 2^-23), and the chunks add in FP32 (about sqrt(300) x 2^-24 over the 300 chunks of a
cluster here): 1.3e-6 with every error at its largest, held to 2e-6, a hundred times less on the
average.  That average is held to 1.25 of the FP32 kernel's.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Operator:
    def __init__(self, imag):
        rng = self.rng = np.random.default_rng(5)
        sizes = rng.integers(30, 65, 64)
        self.off = np.concatenate([[0], np.cumsum(sizes)])
        self.n = n = int(self.off[-1])
        self.M = np.zeros((n, n), np.complex128)
        self.A = np.zeros((2, n, n))                       # moduli: of the products that keep the part of x, and of those that swap it
        self.near, self.far, self.D = [], [], []

        def rand(*s):
            return (rng.normal(size=s) + 1j * imag * rng.normal(size=s)).astype(np.complex64).astype(np.complex128)

        def put(r, c, B, same, swap):
            m, w = B.shape
            self.M[r:r + m, c:c + w] = B
            self.A[0, r:r + m, c:c + w], self.A[1, r:r + m, c:c + w] = same, swap
            if r != c:
                self.M[c:c + w, r:r + m] = B.T
                self.A[0, c:c + w, r:r + m], self.A[1, c:c + w, r:r + m] = same.T, swap.T

        for i, a in enumerate(self.off[:-1]):
            m = int(sizes[i])
            self.D.append(np.diag(rand(m)) + 0j)
            put(a, a, self.D[-1], np.abs(self.D[-1].real), np.abs(self.D[-1].imag))
            for j in range(i + 1, len(sizes)):
                c, w = int(self.off[j]), int(sizes[j])
                if (i + j) % 3:
                    B = rand(m, w)
                    self.near.append((int(a), c, B))
                    put(a, c, B, np.abs(B.real), np.abs(B.imag))
                else:
                    k = int(rng.integers(1, 12))
                    U, V = rand(m, k), rand(k, w)
                    self.far.append((1, int(a), c, U, V))
                    ur, ui, vr, vi = np.abs(U.real), np.abs(U.imag), np.abs(V.real), np.abs(V.imag)
                    put(a, c, U @ V, ur @ vr + ui @ vi, ur @ vi + ui @ vr)

    def handle(self):
        from paper_2307_03968_gb300.hm import HMatrix
        A = HMatrix.from_blocks(np.arange(self.n), self.off, self.D, self.near, self.far)
        A.factor_leaf()
        return A

    def vectors(self, kind, nrhs):
        rng, n = self.rng, self.n
        x = rng.normal(size=(nrhs, n)) + 1j * rng.normal(size=(nrhs, n))
        if kind == "one leaf":
            x *= 2.0 ** -30
            x[:, self.off[7]:self.off[8]] *= 2.0 ** 30
        elif kind == "spread":
            x *= 2.0 ** -rng.uniform(0, 30, size=x.shape)
        elif kind == "real":
            x = x.real + 0j
        return x.astype(np.complex64)

    def errors(self, x, y):
        x = x.astype(np.complex128)
        e = y - x @ self.M.T
        re, im = np.abs(x.real), np.abs(x.imag)
        sr, si = re @ self.A[0].T + im @ self.A[1].T, re @ self.A[1].T + im @ self.A[0].T
        return np.concatenate([(np.abs(e.real) / sr).ravel(), (np.abs(e.imag) / si).ravel()])


@pytest.fixture(scope="module")
def operators():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = {imag: Operator(imag) for imag in (1.0, 2.0 ** -30)}
    held = {imag: o.handle() for imag, o in out.items()}
    yield {imag: (out[imag], held[imag]) for imag in out}
    for A in held.values():
        A.close()


@pytest.mark.parametrize("imag,kind", [(1.0, "even"), (1.0, "one leaf"), (1.0, "spread"), (2.0 ** -30, "real"),
                                       (2.0 ** -30, "even")])
@pytest.mark.parametrize("nrhs", [5, 17, 40, 70])
def test_product_as_accurate_as_fp32(operators, imag, kind, nrhs):
    import torch
    P, A = operators[imag]
    x = P.vectors(kind, nrhs)
    xt = torch.tensor(x, device="cuda")
    yt = torch.empty_like(xt)
    got = {}
    for choice in (16, 32):
        A.set_tuning(nrhs, choice, 0)
        A.apply(xt, yt, n_levels=1, fp64_accumulate=False)
        got[choice] = P.errors(x, yt.cpu().numpy())
    rms = {c: np.sqrt(np.mean(e ** 2)) for c, e in got.items()}
    print("choice 16: rms %.2e max %.2e; 32: rms %.2e max %.2e" % (rms[16], got[16].max(), rms[32], got[32].max()))
    assert got[32].max() < 2e-6
    assert rms[32] <= 1.25 * rms[16]
