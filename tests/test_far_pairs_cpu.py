"""The far-pair route of the mixed form (csrc/farpair.cuh: FP32 corrections around
float-float reference values), compiled for the host, against FP64 quadrature of
the same Gauss points with scipy's Hankel functions.

Bound: FP32 roundings (2^-24) enter through corrections of at most ~0.1 of the
kernel amplitude at k R = 20 and k h <= 0.9, some tens of them per entry, so an
entry is held to 2^-24 of its kernel's amplitude (a quarter of |H| of the pair;
N's 2 x 2 blocks are four times that).  On coarse meshes (k h up to 2.5, where
the route serves pairs beyond zfast only) the corrections reach the size of the
entry and the bound is 2^-19."""

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.special import hankel1

from oracle.geometry import Contour
from oracle.quadrature import gauss_legendre01

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cands = (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc")
    nvcc = next((c for c in cands if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    so = str(tmp_path_factory.mktemp("far") / "far_pairs.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-o", so,
                    os.path.join(HERE, "far_pairs_check.cu")], check=True, capture_output=True, timeout=300)
    return C.CDLL(so)


SHAPES = {"ellipse": dict(ax=1.0, ay=0.5), "superellipse": dict(ax=1.0, ay=0.6, p=4.0),
          "fourier": dict(cos=[1.0, 0.0, 0.004, 0.001], sin=[0.0, 0.0, -0.002, 0.0015])}


@pytest.mark.parametrize("family,N,q,kfac,bits", [("ellipse", 300, 4, 1.0, 24), ("ellipse", 8192, 4, 1.0, 24),
                                                  ("superellipse", 8192, 4, 1.0, 24), ("fourier", 1501, 4, 1.0, 24),
                                                  ("ellipse", 2000, 4, 1.4, 24), ("ellipse", 2000, 3, 1.0, 24),
                                                  ("superellipse", 1000, 6, 1.0, 24), ("ellipse", 2000, 4, 3.9, 19)])
def test_far_pairs_vs_fp64_quadrature(lib, family, N, q, kfac, bits):
    cur = Contour(family, SHAPES[family])
    h, a = cur.L / N, cur.L / (2 * np.pi)
    k = kfac * 2 * np.pi * (N / 10) / cur.L
    beta = 0.4 * k ** (1 / 3) * a ** (-2 / 3)
    kt = k + 1j * beta
    xi, w = gauss_legendre01(q)
    rng = np.random.default_rng(N + q)
    e = rng.integers(0, N, 600)
    f = (e + np.exp(rng.uniform(np.log(20 / kfac), np.log(N / 2), 600)).astype(int)) % N

    def table(el, x):
        s = ((el[:, None] + np.asarray(x)) * h) % cur.L
        p = cur.points(s.ravel())
        return np.ascontiguousarray(np.stack([p[c] for c in ("x", "y", "nx", "ny")], -1).reshape(len(el), -1, 4))

    ce, cg = table(e, [0.5])[:, 0], table(f, [0.5])[:, 0]
    far = k * np.hypot(*(ce - cg)[:, :2].T) >= 20.0 + k * h       # the route's pairs, its nearest included
    e, f, ce, cg = e[far], f[far], np.ascontiguousarray(ce[far]), np.ascontiguousarray(cg[far])
    n = len(e)
    assert n > 100
    pe, pg = table(e, xi), table(f, xi)
    out = np.zeros((n, 6, 4, 2))
    p = lambda v: v.ctypes.data_as(C.c_void_p)   # noqa: E731
    lib.far_pairs(q, p(xi), p(w), C.c_double(k), C.c_double(beta), C.c_double(h), n, p(ce), p(cg), p(pe), p(pg), p(out))
    got = out[..., 0] + 1j * out[..., 1]

    d = pe[:, :, None, :2] - pg[:, None, :, :2]
    R = np.hypot(d[..., 0], d[..., 1])
    g = (d * pg[:, None, :, 2:]).sum(-1) / R
    nd = (pe[:, :, None, 2:] * pg[:, None, :, 2:]).sum(-1)
    ck, ak = np.sqrt(2 / (np.pi * kt)), np.sqrt(2 / (np.pi * k))
    H0, H1, T0, T1 = hankel1(0, k * R) / ak, hankel1(1, k * R) / ak, hankel1(0, kt * R) / ck, hankel1(1, kt * R) / ck
    W = [w * (1 - xi), w * xi]
    gm = -(d * pe[:, :, None, 2:]).sum(-1) / R                  # the mirrored pair's (r' - r).n / R
    amp = [0.25 * np.abs(x).max((1, 2)) for x in (T0, H0, T0)] + [np.abs(H0).max((1, 2))]
    amp += amp[1:3]
    der = np.einsum("p,npr,r->n", w, H0, w)
    for i, K in enumerate((T0, H1 * g, T1 * g, nd * H0, H1 * gm, T1 * gm)):
        for ab in range(4):
            ref = np.einsum("p,npr,r->n", W[ab // 2], K, W[ab % 2])
            if i == 3:
                ref = (der if ab in (0, 3) else -der) - (k * h) ** 2 * ref
            assert np.max(np.abs(got[:, i, ab] - ref) / amp[i]) < 2.0 ** -bits, (i, ab)
