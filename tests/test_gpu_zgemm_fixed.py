"""Complex products through signed 8-bit digits (fxgemm.cu) against extended precision,
entry by entry, with entries of a row and of a column many orders of magnitude apart.

Worst case, a = max_k |A_ik|, b = max_k |B_kj| (componentwise), 2^E <= 2 max per row: with
eight digits a real term errs by 2 (2^-63 2a b) + 7 2^-62 (2a)(2b) < 30 2^-62 a b, 2 k terms:
k a b 2^-55.  Six digits: 2 (2^-47 2a b) + 4 2^-54 (2a)(2b), 2 k terms: k a b 2^-43; plus the
rounding of the result, 2^-51 |C_ij|, in either case.  (The FP32 sums of the lower levels
may add k / 64 times the first bound where all digits are coherent; random ones leave
sqrt(k) 2^-62 a b, which the bound's slack covers.)

Typical case of six digits, on data of one size: A's entries of 24 bits are held exactly, B's
by 2^(E_b - 46) / sqrt(12) rms, and the four dropped digit pairs of a term are products of
two digits of rms 128 / sqrt(3) weighing 2^(E_a + E_b - 68): the error of an entry has

    sigma^2 = 2 k (a_rms^2 2^(2 E_b - 92) / 12 + 4 (128^2 / 3)^2 2^(2 (E_a + E_b) - 136)),

and 13 000 of them stay within 8 sigma.  (One more dropped level would be sixteen times the
pairs' part: 9 sigma rms.)"""

import numpy as np
import pytest

from gpu_common import built, to_np

pytestmark = pytest.mark.gpu


def crandn(g, *shape):
    return g.standard_normal(shape) + 1j * g.standard_normal(shape)


def bf16_planes(x):
    """Sum of the three bf16 planes of x (real): each the remainder rounded to 8 bits, half to even."""
    total, r = np.zeros_like(x), x.copy()
    for _ in range(3):
        m, e = np.frexp(r)
        p = np.ldexp(np.rint(m * 256.0) / 256.0, e)
        total, r = total + p, r - p
    return total


def cmax(X, axis):
    return np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis=axis, keepdims=True)


def product(A, B, add=None):
    # (numpy has no fast extended-precision product: real ones of the parts)
    L = np.longdouble
    re = A.real.astype(L) @ B.real.astype(L) - A.imag.astype(L) @ B.imag.astype(L)
    im = A.real.astype(L) @ B.imag.astype(L) + A.imag.astype(L) @ B.real.astype(L)
    if add is not None:
        re, im = re + add.real, im + add.imag
    return re, im


def errors(got, ref):
    return np.maximum(np.abs(got.real - ref[0]), np.abs(got.imag - ref[1])).astype(float)


# around the tile of 128 rows and 32 columns, the stage of 16 and the chunk of 64 complex K-values
SIZES = [(1, 1, 1), (128, 32, 64), (129, 33, 65), (300, 43, 391), (257, 7, 1030)]


@pytest.mark.parametrize("m,n,k", SIZES)
@pytest.mark.parametrize("digits,bits", [(8, 55), (6, 43)])
@pytest.mark.parametrize("spread", [0.0, 8.0])
def test_worst_case_bound(m, n, k, digits, bits, spread):
    built()
    from paper_2203_13283_gb300.solver import zgemm_fixed
    g = np.random.default_rng(m + n + k + digits)
    A = crandn(g, m, k) * 10.0 ** g.uniform(-spread, 0, (m, k)) * 10.0 ** g.uniform(-3, 3, (m, 1))
    B = crandn(g, k, n) * 10.0 ** g.uniform(-spread, 0, (k, n)) * 10.0 ** g.uniform(-6, 6, (1, n))
    add = crandn(g, m, n) * cmax(A, 1) * cmax(B, 0)
    stored = bf16_planes(A.real) + 1j * bf16_planes(A.imag) if digits == 6 else A
    for c in (None, add):
        got, ref = to_np(zgemm_fixed(A, B, c, digits)), product(stored, B, c)
        size = np.maximum(np.abs(ref[0]), np.abs(ref[1])).astype(float)
        bound = k * cmax(stored, 1) * cmax(B, 0) * 2.0 ** -bits + 2.0 ** -51 * size
        assert np.all(errors(got, ref) <= bound)


@pytest.mark.parametrize("m,n,k", [(301, 43, 391), (130, 100, 2000)])
def test_six_digits_on_data_of_one_size(m, n, k):
    built()
    from paper_2203_13283_gb300.solver import zgemm_fixed
    g = np.random.default_rng(k)
    A = crandn(g, m, k) * 2.0 ** g.integers(-9, 9, (m, 1))
    B = crandn(g, k, n) * 2.0 ** g.integers(-20, 20, (1, n))
    stored = bf16_planes(A.real) + 1j * bf16_planes(A.imag)
    ref = product(stored, B)
    ea, eb = (np.frexp(cmax(X, ax))[1].astype(float) for X, ax in ((stored, 1), (B, 0)))
    a_rms = np.sqrt(np.mean(np.abs(A) ** 2, axis=1, keepdims=True) / 2)
    sigma = np.sqrt(2 * k * (a_rms ** 2 * 4.0 ** (eb - 46) / 12 + 4 * (128.0 ** 2 / 3) ** 2 * 4.0 ** (ea + eb - 68)))
    err = errors(to_np(zgemm_fixed(A, B, digits=6)), ref)
    size = np.maximum(np.abs(ref[0]), np.abs(ref[1])).astype(float)
    assert np.all(err <= 8 * sigma + 2.0 ** -51 * size), np.max(err / sigma)


@pytest.mark.parametrize("m,n", [(300, 100), (128, 33), (129, 32)])
def test_panels_give_the_values_of_one(m, n):
    """Operands in panels of one tile each (128 rows, 32 columns), K of one chunk: the same
    sums, with and without an addend."""
    built()
    from paper_2203_13283_gb300.solver import zgemm_fixed
    g = np.random.default_rng(m * n)
    A, B, add = crandn(g, m, 60), crandn(g, 60, n), crandn(g, m, n)
    for c in (None, add):
        assert np.array_equal(to_np(zgemm_fixed(A, B, c, panel_bytes=1)), to_np(zgemm_fixed(A, B, c)))


def test_panels_of_long_rows():
    built()
    from paper_2203_13283_gb300.solver import zgemm_fixed
    g = np.random.default_rng(9)
    A, B, add = crandn(g, 300, 1500), crandn(g, 1500, 70), crandn(g, 300, 70)
    got, ref = to_np(zgemm_fixed(A, B, add, panel_bytes=1)), product(A, B, add)
    size = np.maximum(np.abs(ref[0]), np.abs(ref[1])).astype(float)
    assert np.all(errors(got, ref) <= 1500 * cmax(A, 1) * cmax(B, 0) * 2.0 ** -55 + 2.0 ** -51 * size)
