"""Kernels that split a transform, a filter or a sum over CTAs by rules on sizes: both
sides of each rule and the ragged sizes, against numpy or the FP64 form.

Bounds.  FP64 results: a few hundred roundings of 2^-53 at most, amplified by the
cyclic Gram matrix's condition (3) where it is inverted: 1e-12.  Mixed form: the form's
own bar for an operator product (2e-6 per column); its circulant applies for N not a
power of two stay FP64 transforms, as convolutions with the inverse transform of mu_C,
whose FP64 rounding grows with mu_C's spread (below 1e3 here): 2e-12, the bar of the
transform of any length.  Far field: FP64 sums over the same quadrature points, whose
positions the library finds by FP64 arc-length inversion (~1e-12): 1e-9."""

import functools

import numpy as np
import pytest
import torch

from gpu_common import colrel, make_solver, to_np

pytestmark = pytest.mark.gpu

ELL = dict(family="ellipse", params={"ax": 1.0, "ay": 0.5})


def randn(N, B, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(N, B, dtype=torch.complex128, device="cuda", generator=g)


@functools.lru_cache(maxsize=1)
def assembled(N, mixed):
    s = make_solver(dict(ELL, N=N, k=None), precision=int(mixed))
    s.assemble()
    return s


# one chunk shorter than the filter's warm-up, full and short last chunks, the largest
# column of one CTA (2048), one beyond it (last chunk of one sample, of 52, full)
@pytest.mark.parametrize("N", [12, 39, 64, 65, 127, 1000, 2048, 2049, 2100, 4096])
def test_gram_inverse(N):
    s = assembled(N, False)
    X = randn(N, 3)
    lam = (4.0 + 2.0 * np.cos(2.0 * np.pi * np.arange(N) / N)) * (s.info()["h"] / 6.0)
    want = np.fft.ifft(np.fft.fft(to_np(X), axis=0) / lam[:, None], axis=0)
    assert colrel(to_np(s.apply("GINV", X)), want) < 1e-12
    # in place: the same values on either route
    Y = X.t().contiguous()
    lib, ptr = s.lib, Y.data_ptr()
    assert lib.wcs_apply(s.h, 11, 3, ptr, N, ptr, N) == 0
    assert torch.equal(Y.t(), s.apply("GINV", X))


# on both sides of the one kernel's range: 16384 chunks of 64 samples (256 columns of 64
# chunks, 496 of 33) and 2560 CTAs; every column has the values that it has by itself
@pytest.mark.parametrize("N, B", [(64, 2560), (64, 2561), (4096, 256), (4096, 257), (2100, 496), (2100, 497)])
def test_gram_inverse_of_many_columns(N, B):
    s = assembled(N, False)
    X = randn(N, B)
    Y = s.apply("GINV", X)
    for c in (0, B // 2, B - 1):
        assert torch.equal(Y[:, c:c + 1], s.apply("GINV", X[:, c:c + 1])), c


# lengths on both sides of the two-half transform's range, column counts on both sides
# of its limit
@pytest.mark.parametrize("N", [256, 512, 1024, 4096, 8192])
@pytest.mark.parametrize("B", [1, 3, 76, 77])
def test_fp64_circulant_columns(N, B):
    s = assembled(N, False)
    X = randn(N, B)
    mu = to_np(s.circulant_eigs("CC"))[:, None]
    f = np.fft.fft(to_np(X), axis=0)
    assert colrel(to_np(s.apply("CC", X)), np.fft.ifft(mu * f, axis=0)) < 1e-12
    assert colrel(to_np(s.apply("CC_INV", X)), np.fft.ifft(f / mu, axis=0)) < 1e-12


@pytest.mark.parametrize("N", [97, 600, 1025, 2777])
@pytest.mark.parametrize("B", [1, 5, 40])
def test_mixed_products_and_convolutions(N, B):
    s = assembled(N, True)
    X = randn(N, B)
    x = to_np(X)
    mu = to_np(s.circulant_eigs("CC"))[:, None]
    f = np.fft.fft(x, axis=0)
    for op, m in (("CC", mu), ("CCH", mu.conj()), ("CC_INV", 1 / mu), ("CCH_INV", 1 / mu.conj())):
        assert colrel(to_np(s.apply(op, X)), np.fft.ifft(m * f, axis=0)) < 2e-12, op
    # C and C^H from the four operators, the Gram filters in FP64 on the host
    h = s.info()["h"]
    lam = ((4.0 + 2.0 * np.cos(2.0 * np.pi * np.arange(N) / N)) * (h / 6.0))[:, None]

    def gram(v, inverse=False):
        return np.fft.ifft(np.fft.fft(v, axis=0) * (1 / lam if inverse else lam), axis=0)

    def mul(op, v):
        return to_np(s.apply(op, torch.as_tensor(np.ascontiguousarray(v), device="cuda")))

    t1 = gram(0.5 * gram(x) - mul("D", x), True)
    t2 = gram(mul("N", x), True)
    want = 0.5 * gram(t1) + mul("DT", t1) + mul("S", t2)
    assert colrel(to_np(s.apply("C", X)), want) < 2e-6
    # <y, C x> = <C^H y, x>
    y = randn(N, B, 1)
    lhs = np.sum(to_np(y).conj() * want, axis=0)
    rhs = np.sum(to_np(s.apply("CH", y)).conj() * x, axis=0)
    scale = np.linalg.norm(to_np(y), axis=0) * np.linalg.norm(want, axis=0)
    assert np.max(np.abs(lhs - rhs) / scale) < 2e-6


# the near band, the tabulated Hankel functions and the far tiles meet in every row:
# rows of the assembled planes against the entries integrated one by one in FP64
@pytest.mark.parametrize("N,options", [(61, {}), (200, {}), (401, dict(q_far=3, q_near=9)), (333, dict(zfast=9.0))])
def test_mixed_rows_vs_entries(N, options):
    s = make_solver(dict(ELL, N=N, k=None), precision=1, **options)
    s.assemble()
    cols = np.unique([0, 1, N // 3, N - 2, N - 1])
    eye = torch.zeros(N, len(cols), dtype=torch.complex128, device="cuda")
    eye[torch.as_tensor(cols), torch.arange(len(cols))] = 1.0
    r, c = np.meshgrid(np.arange(N), cols, indexing="ij")
    want = s.operator_entries(r.ravel(), c.ravel())
    for op, key in (("S", "S"), ("D", "D"), ("DT", "Dt"), ("N", "N")):
        got = to_np(s.apply(op, eye))
        assert colrel(got, want[key].reshape(N, len(cols))) < 2e-6, op
    s.close()


@pytest.mark.parametrize("N,kh,q,nphi", [(97, 0.85, 8, 1), (130, 0.63, 16, 33), (64, 0.2, 5, 31), (65, 0.89, 7, 32),
                                         (203, 0.89, 4, 100), (90, 0.95, 8, 40)])
def test_farfield_map(N, kh, q, nphi):
    s = make_solver(dict(ELL, N=N, k=1.0), q_near=q)
    k = kh / s.info()["h"]
    s.mesh(N, k)
    h = s.info()["h"]
    x, w = np.polynomial.legendre.leggauss(q)
    x, w = (x + 1) / 2, w / 2
    g = s.geometry_sample(((np.arange(N)[:, None] + x) * h).ravel())
    J = randn(N, 4)
    j = to_np(J)
    phi = np.arange(nphi) * 0.7 + 0.1
    rise = np.repeat(np.roll(j, -1, axis=0), q, axis=0)   # element e carries hats e (falling) and e + 1 (rising)
    fall = np.repeat(j, q, axis=0)
    xs, ws = np.tile(x, N)[:, None], np.tile(w, N)[:, None] * h
    cur = ws * ((1 - xs) * fall + xs * rise)
    d = np.cos(phi)[:, None] * g["x"] + np.sin(phi)[:, None] * g["y"]
    n = np.cos(phi)[:, None] * g["nx"] + np.sin(phi)[:, None] * g["ny"]
    want = 1j * k * np.exp(0.25j * np.pi) / np.sqrt(8 * np.pi * k) * ((n * np.exp(-1j * k * d)) @ cur)
    assert colrel(to_np(s.farfield(J, phi)), want) < 1e-9
    s.close()


def test_capacitance_inverse_beyond_a_block():
    # rank above one block's 256 rows: the Woodbury inverse against the matrix it
    # inverts, C_c + U V^T, whatever the skeleton left out of C.  Gauss-Jordan with
    # partial pivoting: r 2^-53 cond(K) ~ 300 * 1e-16 * 1e4 = 3e-10; 1e-8 allows for
    # pivot growth
    N = 700
    s = make_solver(dict(ELL, N=N, k=None))
    s.assemble()
    assert s.skeleton(1e-14, max_rank=300, seed=3, allow_cap=True) > 256
    s.factor()
    b = randn(N, 3)
    x = s.woodbury_apply(b)
    assert colrel(to_np(s.apply("CC", x)) + to_np(s.apply("SKEL", x)), to_np(b)) < 1e-8
    s.close()
