"""The FP64 division, reciprocal and square root of fp64_math.cuh against IEEE
arithmetic (numpy's and CUDA's operators): random mantissas and exponents, mantissas
next to powers of two and to 3/2, and arguments around the range switches.

Bounds: the reciprocal's series leaves 2^-72, so its last rounding decides: 0.5 ulp and
a 2^-18 of one. Quotients and roots are the rounded ones but where they lie within
2^-50 ulp of the middle of two numbers (next to powers of two some do), that is, within
0.5 ulp and a 2^-50 of one. The power x^-a, a = k / n, against 50 decimal digits: the
first term left out of the series is 2^-56 relative (0.08 ulp). At n = 3 the rounding of
one product and the last one remain, at n = 2 these at most, at other n those of up to
five products with weights of at most one, half an ulp each; its reciprocal 1 / x leaves
2^-58. Without a plan it is pow, which CUDA documents at 2 ulp."""
import subprocess
from decimal import Decimal, localcontext
from fractions import Fraction

import numpy as np
import pytest

from paper_2107_01664_gb300 import build

pytestmark = pytest.mark.gpu
N = 1 << 17


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import os
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("fp64")
    src = os.path.join(os.path.dirname(__file__), "fp64_math_driver.cu")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-I", build.CSRC, "-o", str(d / "drv"), src],
                   check=True)

    def run(op, a, b=None):
        b = np.ones_like(a) if b is None else b
        with open(d / "in", "wb") as f:
            np.array([op, len(a)], np.int32).tofile(f)
            a.tofile(f)
            b.tofile(f)
        subprocess.run([str(d / "drv"), str(d / "in"), str(d / "out")], check=True)
        out = np.fromfile(d / "out", np.float64)
        return out[:len(a)], out[len(a):]

    return run


def numbers(seed, lo, hi, n=N):
    """n numbers with exponents in [lo, hi): random mantissas, then edge mantissas."""
    rng = np.random.default_rng(seed)
    m = 1.0 + rng.random(n)
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 1.5 - 2.0 ** -52, 1.5 + 2.0 ** -52])
    m[::8] = edge[rng.integers(0, len(edge), len(m[::8]))]
    return np.ldexp(m, rng.integers(lo, hi, n).astype(np.int32)) * rng.choice([-1.0, 1.0], n)


def split(x):
    c = 134217729.0 * x
    h = c - (c - x)
    return h, x - h


def rounded(x, want, exact):
    """x is `want`, the rounded result, or as near to exact(i), to a 2^-50 of an ulp."""
    for i in np.flatnonzero(x != want):
        ulp = Fraction(float(np.spacing(abs(want[i]))))
        if abs(Fraction(float(x[i])) - exact(i)) > (Fraction(1, 2) + Fraction(1, 2 ** 50)) * ulp:
            return False
    return True


def reciprocal_error(x, y):
    """(y - 1 / x) in ulps of y, to 2^-40: the product x y exactly as a sum of two."""
    m, e = np.frexp(x)
    x, y = m, np.ldexp(y, e)              # x in [1/2, 1): nothing over- or underflows
    p = x * y
    (xh, xl), (yh, yl) = split(x), split(y)
    r = ((xh * yh - p) + xh * yl + xl * yh) + xl * yl
    return ((p - 1.0) + r) / x / np.spacing(np.abs(y))


@pytest.mark.parametrize("lo,hi", [(-1, 2), (-60, 60), (-1000, 1000)])
def test_reciprocal(call, lo, hi):
    x = numbers(1, lo, hi)
    y, cuda = call(0, x)
    assert np.abs(reciprocal_error(x, y)).max() <= 0.5 + 2.0 ** -18
    assert np.array_equal(cuda, 1.0 / x)


@pytest.mark.parametrize("lo,hi", [(-1, 2), (-60, 60), (-900, 900)])
def test_quotient(call, lo, hi):
    b = numbers(2, lo, hi)
    q = numbers(3, max(lo, -60), min(hi, 60))
    a = b * q
    x, cuda = call(1, a, b)
    assert np.array_equal(cuda, a / b)
    assert rounded(x, cuda, lambda i: Fraction(float(a[i])) / Fraction(float(b[i])))
    assert np.array_equal(call(1, np.zeros(4), b[:4])[0], np.zeros(4))


@pytest.mark.parametrize("lo,hi", [(-1, 2), (-60, 60), (-1000, 1000), (-935, -925), (925, 935)])
def test_root_and_its_reciprocal(call, lo, hi):      # 2^930 = 1e280: the switch to sqrt()
    x = np.abs(numbers(4, lo, hi))
    s, r = call(2, x)
    # (Newton's step from s - 1 ulp .. s + 1 ulp on the root to 2^-100)
    assert rounded(s, np.sqrt(x), lambda i: (lambda v, w: (w + v / w) / 2)(Fraction(float(x[i])),
                                                                           Fraction(float(s[i]))))
    assert np.abs(reciprocal_error(s, r)).max() <= 0.5 + 2.0 ** -18


def test_third(call):
    x = numbers(5, -900, 900)
    y, cuda = call(3, x)
    assert np.array_equal(cuda, x / 3.0)
    assert rounded(y, cuda, lambda i: Fraction(float(x[i])) / 3)


@pytest.mark.parametrize("p,kn,kl", [(6.0, (3, 5), (3, 4)), (3.0, (3, 4), (3, 5)), (4.5, (9, 14), (9, 13)),
                                     (4.0, (2, 3), (2, 3)), (5.0, (5, 8), (5, 7)), (2.5, (5, 6), (5, 9)),
                                     (32.0 / 13.0, (16, 19), (16, 29)), (3.7, None, None)])
@pytest.mark.parametrize("low", [False, True])
@pytest.mark.parametrize("lo,hi", [(-3, 3), (-40, 20), (-100, 100), (-140, -100), (100, 140)])
def test_rational_power(call, p, kn, kl, low, lo, hi):      # 2^-100 .. 2^100: the plan's range
    x = np.abs(numbers(6, lo, hi, 1500))
    b = np.full_like(x, -p if low else p)
    y, ix = call(4, x, b)
    n, k = (kl if low else kn) or (0, 0)
    a = float(call(5, x, b)[1][0])
    with localcontext() as c:
        c.prec = 50
        e = Decimal(k) / Decimal(n) if n else Decimal(a)
        want = [(-e * Decimal(float(v)).ln()).exp() for v in x]
        err = np.array([abs(float((Decimal(float(u)) - w) / Decimal(float(np.spacing(u))))) for u, w in zip(y, want)])
        inv = np.array([abs(float((Decimal(float(u)) - 1 / Decimal(float(v))) / Decimal(float(np.spacing(u)))))
                        for u, v in zip(ix, x)])
    # outside its range, and without a plan, pow to the rounded exponent a: a's own rounding
    # (2^-54 a) adds 2^-54 a |ln x| relative
    plan = n > 0 and -100 <= lo and hi <= 100
    bound = (1.08 if n <= 3 else 3.08) if plan else 2.0 + a * np.abs(np.log(x))
    assert np.all(err <= bound), err.max()
    assert inv.max() <= 0.53
