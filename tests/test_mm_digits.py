"""Exact model of the matrix-instruction residual's arithmetic (csrc/k_mm.cu) in numpy float32, whose
operations round as the kernel's do: the digits of an operand and what they leave out, the size of
a chunk's digit sums, and the short form of TwoSum that joins them.
"""

import numpy as np
import pytest

f = np.float32
MAGIC = f(12582912.0)                                      # 1.5 x 2^23: adding and taking it off rounds to an integer


def nearest(v):
    return (v + MAGIC) - MAGIC


def digits(v, lo):
    t = v * f(256)
    d = [nearest(t)]
    t = (t - d[0]) * f(512)
    d.append(nearest(t))
    t = (t - d[1]) * f(512)
    low = lo * f(67108864)
    d.append(nearest(t + low))
    t = ((t - d[2]) + low) * f(512)
    d.append(nearest(t))
    d.append((t - d[3]) * f(512))
    return d


WEIGHTS = [2.0 ** -8, 2.0 ** -17, 2.0 ** -26, 2.0 ** -35, 2.0 ** -44]


def operands(kind, n=200000):
    rng = np.random.default_rng(1)
    v = rng.uniform(-1, 1, n)
    if kind == "graded":
        v *= 2.0 ** -rng.uniform(0, 40, n)
    elif kind == "edges":                                  # halves and carries of the digits, and the scale itself
        v = rng.integers(-512, 513, n) / 512 + rng.integers(-2, 3, n) * 2.0 ** -rng.integers(9, 40, n)
        v = np.clip(v, -1, 1)
    hi = v.astype(f)
    lo = (rng.uniform(-0.5, 0.5, n) * np.spacing(np.abs(hi))).astype(f)
    return hi, lo


@pytest.mark.parametrize("kind", ["even", "graded", "edges"])
@pytest.mark.parametrize("trailing", [False, True])
def test_digits_hold_the_operand(kind, trailing):
    hi, lo = operands(kind)
    if not trailing:
        lo = np.zeros_like(lo)
    d = digits(hi, lo)
    for q in d[:4]:
        assert np.all(q == np.rint(q)) and np.abs(q).max() <= 258
        assert np.all(q.astype(np.float16).astype(f) == q)     # held exactly by FP16
    assert np.abs(d[4]).max() <= 257
    rest = d[4].astype(np.float16).astype(np.float64)
    got = sum(w * q.astype(np.float64) for w, q in zip(WEIGHTS, d[:4])) + WEIGHTS[4] * rest
    off = np.abs(got - (hi.astype(np.float64) + lo.astype(np.float64)))
    assert off.max() <= 2.0 ** -46 if trailing else off.max() <= 2.0 ** -48
    if not trailing:                                       # an FP32 operand within 2^24 of the scale: exactly
        assert np.all(off[np.abs(hi) >= 2.0 ** -24] == 0)


def test_chunk_sums_are_exact_integers():
    # up to four digit products a sum, 16 K, real and imaginary part: 4 x 32 products of 258 x 258 at most
    assert 4 * 32 * 258 * 258 < 2 ** 24


def short_two_sum(a, b, weight):
    """s + e for a + weight b as the kernel forms them: fma, sub, fma (the product weight b is exact)."""
    wb = b.astype(np.float64) * weight
    s = (a.astype(np.float64) + wb).astype(f)
    e = (wb + (a - s).astype(np.float64)).astype(f)
    return s, e


def test_short_two_sum_is_exact():
    rng = np.random.default_rng(2)
    n = 400000

    def sums(most):                                        # integers of every size up to the largest sum, zero among them
        v = np.rint(rng.uniform(-1, 1, n) * most * 2.0 ** -rng.uniform(0, 24, n))
        v[::17] = 0
        return v.astype(f)

    h0, h1, h2 = sums(32 * 2 ** 16), sums(2 * 32 * 2 ** 16), sums(3 * 32 * 2 ** 16)
    s, e = short_two_sum(h0, h1, 2.0 ** -9)
    assert np.all(s.astype(np.float64) + e == h0.astype(np.float64) + h1 * 2.0 ** -9)
    v, e2 = short_two_sum(s, h2, 2.0 ** -18)
    assert np.all(v.astype(np.float64) + e2 == s.astype(np.float64) + h2 * 2.0 ** -18)
