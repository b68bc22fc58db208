"""Routes that are chosen by sizes and options, on the sides that the other tests leave out:
coarse meshes (k h above 0.9), near bands of other widths, transforms of more columns than a
plan's work holds, convolutions whose transforms go through memory twice, the circle's
eigenvalues from tabulated Hankel functions.

Bounds.  An operator's column against entries integrated one by one by the general FP64 path:
the same rule, other sums; 1e-12 in the FP64 form, the mixed form's bar for an operator product
(2e-6 per column) there.  Circulant applies: 1e-12 (FP64 form), 2e-12 (mixed form, whose
inverse transform of mu_C enters).  Eigenvalues: N entries of relative error ~1e-15 at most
each (the table's interpolation, below 1e-16, and roundings of ~10 operations a point), summed
by an FP64 transform: 1e-13 of the largest; for N, whose entries are differences of terms of
a quarter of |H0| each, 1e-15 of the sum of its terms."""

import numpy as np
import pytest
import torch
from scipy.special import hankel1

from gpu_common import colrel, make_solver, to_np

pytestmark = pytest.mark.gpu

ELL = dict(family="ellipse", params={"ax": 1.0, "ay": 0.5})


def randn(N, B, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(N, B, dtype=torch.complex128, device="cuda", generator=g)


def check_columns(s, tol):
    N = s.N
    cols = np.unique([0, 1, N // 3, N // 2 + 1, N - 2, N - 1])
    eye = torch.zeros(N, len(cols), dtype=torch.complex128, device="cuda")
    eye[torch.as_tensor(cols), torch.arange(len(cols))] = 1.0
    r, c = np.meshgrid(np.arange(N), cols, indexing="ij")
    want = s.operator_entries(r.ravel(), c.ravel())
    for op, key in (("S", "S"), ("D", "D"), ("DT", "Dt"), ("N", "N")):
        assert colrel(to_np(s.apply(op, eye)), want[key].reshape(N, len(cols))) < tol, op


@pytest.mark.parametrize("N", [97, 500])
@pytest.mark.parametrize("kh", [0.91, 1.5, 2.4])
@pytest.mark.parametrize("options", [dict(precision=0), dict(precision=1), dict(precision=1, zfast=0.0),
                                     dict(precision=1, zfast=40.0)])
def test_coarse_meshes(N, kh, options):
    s = make_solver(dict(ELL, N=N, k=None), **options)
    s.mesh(N, kh / s.info()["h"])
    s.assemble()
    check_columns(s, 2e-6 if options["precision"] else 1e-12)
    s.close()


# a band of one element, wider ones, one as wide as a tile, one that covers the contour
@pytest.mark.parametrize("N,band", [(200, 1), (333, 2), (200, 7), (333, 33), (61, 30), (61, 40)])
@pytest.mark.parametrize("precision", [0, 1])
def test_near_bands(N, band, precision):
    s = make_solver(dict(ELL, N=N, k=None), precision=precision, near_band=band)
    s.assemble()
    check_columns(s, 2e-6 if precision else 1e-12)
    s.close()


@pytest.mark.parametrize("N", [12, 13, 20, 60])
@pytest.mark.parametrize("options", [dict(precision=0), dict(precision=1), dict(precision=1, near_band=6)])
def test_small_k_a(N, options):
    """k~ off the tables' form (Im k~ above a tenth of k): near bands by the full expansions, or,
    where they cover the contour, pair by pair."""
    s = make_solver(dict(ELL, N=N, k=None), **options)
    i = s.info()
    assert i["kt_im"] > 0.1 * i["k"]
    s.assemble()
    check_columns(s, 2e-6 if options["precision"] else 1e-12)
    s.close()


def test_coarse_mesh_with_a_sorted_band():
    # k h (near_band + 1) below 3.9: the FP64 form's sorted pairs on a coarse mesh
    s = make_solver(dict(ELL, N=300, k=None), near_band=1)
    s.mesh(300, 1.7 / s.info()["h"])
    s.assemble()
    check_columns(s, 1e-12)
    s.close()


# a plan's work holds 256 columns; a pass more than its scratch takes one CTA a column
@pytest.mark.parametrize("N", [512, 600, 4096])
@pytest.mark.parametrize("B", [256, 257, 300])
def test_circulant_columns_around_a_plans_work(N, B):
    s = make_solver(dict(ELL, N=N, k=None), rhs_chunk=512)
    s.assemble()
    X = randn(N, B)
    mu, f = to_np(s.circulant_eigs("CC"))[:, None], np.fft.fft(to_np(X), axis=0)
    assert colrel(to_np(s.apply("CC", X)), np.fft.ifft(mu * f, axis=0)) < 1e-12
    assert colrel(to_np(s.apply("CC_INV", X)), np.fft.ifft(f / mu, axis=0)) < 1e-12
    s.close()


# two transforms of 8192, three of 8192, two of 16384 points
@pytest.mark.parametrize("N", [6200, 9001, 13000])
def test_convolutions_of_long_transforms(N):
    s = make_solver(dict(ELL, N=N, k=None), precision=1)
    s.assemble()
    X = randn(N, 5)
    mu, f = to_np(s.circulant_eigs("CC"))[:, None], np.fft.fft(to_np(X), axis=0)
    for op, m in (("CC", mu), ("CCH", mu.conj()), ("CC_INV", 1 / mu), ("CCH_INV", 1 / mu.conj())):
        assert colrel(to_np(s.apply(op, X)), np.fft.ifft(m * f, axis=0)) < 2e-12, op
    s.close()


@pytest.mark.parametrize("N", [97, 512, 4099])
@pytest.mark.parametrize("kh", [None, 0.3, 1.5])
def test_circle_eigenvalues_of_both_forms(N, kh):
    """The same rules: tabulated Hankel functions below k R = 24 (mixed form), full expansions."""
    mu = []
    for precision in (1, 0):
        s = make_solver(dict(ELL, N=N, k=None), precision=precision, q_far=4, q_near=8)
        if kh:
            s.mesh(N, kh / s.info()["h"])
        s.assemble()
        i = s.info()
        mu.append({op: to_np(s.circulant_eigs(op)) for op in ("S", "D", "DT", "N")})
        s.close()
    for op in ("S", "D", "DT"):
        assert np.max(np.abs(mu[0][op] - mu[1][op])) < 1e-13 * np.max(np.abs(mu[1][op])), op
    # N: the four element pairs of an entry cancel to ~(k h)^2 of a term (Maue's form)
    R = np.maximum(2.0 * i["a"] * np.sin(np.pi * np.arange(N) / N), 0.5 * i["h"])
    terms = np.sum(np.abs(hankel1(0, i["k"] * R)))
    assert np.max(np.abs(mu[0]["N"] - mu[1]["N"])) < 1e-15 * terms


# both sides of the map's rule (16 angles, 65536 of N times angles), meshes and rules of the moments
@pytest.mark.parametrize("N,nphi,kh,q", [(12, 1, 0.63, 8), (63, 100, 0.63, 8), (1023, 64, 0.63, 8), (1024, 64, 0.63, 8),
                                         (4400, 15, 0.63, 8), (4097, 16, 0.63, 8), (730, 90, 0.89, 4), (2200, 33, 0.85, 16),
                                         (301, 219, 0.2, 5), (911, 73, 0.89, 7)])
def test_farfield_map_around_its_rule(N, nphi, kh, q):
    """Against the same quadrature in numpy (positions from the library's arc-length inversion,
    ~1e-12: 1e-9)."""
    s = make_solver(dict(ELL, N=N, k=None), q_near=q)
    s.mesh(N, kh / s.info()["h"])
    i = s.info()
    k, h = i["k"], i["h"]
    x, w = np.polynomial.legendre.leggauss(q)
    x, w = (x + 1) / 2, w / 2
    g = s.geometry_sample(((np.arange(N)[:, None] + x) * h).ravel())
    J = randn(N, 4)
    j = to_np(J)
    phi = np.arange(nphi) * 0.7 + 0.1
    cur = np.tile(w, N)[:, None] * h * (np.tile(1 - x, N)[:, None] * np.repeat(j, q, axis=0)
                                        + np.tile(x, N)[:, None] * np.repeat(np.roll(j, -1, axis=0), q, axis=0))
    d = np.cos(phi)[:, None] * g["x"] + np.sin(phi)[:, None] * g["y"]
    n = np.cos(phi)[:, None] * g["nx"] + np.sin(phi)[:, None] * g["ny"]
    want = 1j * k * np.exp(0.25j * np.pi) / np.sqrt(8 * np.pi * k) * ((n * np.exp(-1j * k * d)) @ cur)
    assert colrel(to_np(s.farfield(J, phi)), want) < 1e-9
    s.close()
