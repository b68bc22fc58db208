"""The far-pair route on elements that turn sharply: ellipses whose tips turn by up to a
radian within an element, where the route is still taken.  As in test_far_pairs_cpu.py an
entry is held to 2^-24 of its kernel's amplitude, against FP64 quadrature of the same points
with scipy's Hankel functions."""

import ctypes as C

import numpy as np
import pytest
from scipy.special import ellipe, ellipeinc, hankel1

from oracle.quadrature import gauss_legendre01
from test_far_pairs_cpu import lib  # noqa: F401


def ellipse_points(b, s):
    """x, y, nx, ny at arc lengths s of x^2 + y^2 / b^2 = 1, counter-clockwise from (1, 0)."""
    m, quarter = 1.0 - b * b, ellipe(1.0 - b * b)
    # arc length from (0, b): ellipeinc(t, m) at (sin t, b cos t); counter-clockwise from (1, 0) t falls from pi / 2
    t = 0.5 * np.pi - s / quarter * 0.5 * np.pi
    for _ in range(60):
        t = t - np.clip((ellipeinc(t, m) - (quarter - s)) / np.sqrt(1.0 - m * np.sin(t) ** 2), -0.3, 0.3)
    x, y = np.sin(t), b * np.cos(t)
    n = np.hypot(b * x, y / b)
    return np.stack([x, y, b * x / n, y / b / n], -1)


@pytest.mark.parametrize("b,N,kh", [(0.05, 1610, 0.63), (0.05, 1610, 0.9), (0.1, 410, 0.63), (0.1, 410, 0.9), (0.2, 150, 0.9)])
def test_sharply_curved_elements(lib, b, N, kh):  # noqa: F811
    L, q = 4.0 * ellipe(1.0 - b * b), 4
    h, a = L / N, L / (2 * np.pi)
    k = kh / h
    assert h / b ** 2 <= 1.0 and (b == 0.2 or h / b ** 2 > 0.95)
    beta = 0.4 * k ** (1 / 3) * a ** (-2 / 3)
    kt = k + 1j * beta
    xi, w = gauss_legendre01(q)
    at = lambda x: ellipse_points(b, (np.arange(N)[:, None] + np.asarray(x)) * h)   # noqa: E731
    P, cen = at(xi), at([0.5])[:, 0]
    rng = np.random.default_rng(N)
    tips = np.concatenate([np.arange(-4, 5) % N, (N // 2 + np.arange(-4, 5)) % N])
    e = np.concatenate([rng.choice(tips, 1500), rng.integers(0, N, 500)])
    f = rng.integers(0, N, 2000)
    far = k * np.hypot(*(cen[e] - cen[f])[:, :2].T) >= 20.0 + kh
    e, f = e[far], f[far]
    n = len(e)
    assert n > 500
    pe, pg, ce, cg = (np.ascontiguousarray(v) for v in (P[e], P[f], cen[e], cen[f]))
    out = np.zeros((n, 6, 4, 2))
    p = lambda v: v.ctypes.data_as(C.c_void_p)   # noqa: E731
    lib.far_pairs(q, p(xi), p(w), C.c_double(k), C.c_double(beta), C.c_double(h), n, p(ce), p(cg), p(pe), p(pg), p(out))
    got = out[..., 0] + 1j * out[..., 1]
    d = pe[:, :, None, :2] - pg[:, None, :, :2]
    R = np.hypot(d[..., 0], d[..., 1])
    g = (d * pg[:, None, :, 2:]).sum(-1) / R
    gm = -(d * pe[:, :, None, 2:]).sum(-1) / R
    nd = (pe[:, :, None, 2:] * pg[:, None, :, 2:]).sum(-1)
    ck, ak = np.sqrt(2 / (np.pi * kt)), np.sqrt(2 / (np.pi * k))
    H0, H1, T0, T1 = hankel1(0, k * R) / ak, hankel1(1, k * R) / ak, hankel1(0, kt * R) / ck, hankel1(1, kt * R) / ck
    W = [w * (1 - xi), w * xi]
    amp = [0.25 * np.abs(x).max((1, 2)) for x in (T0, H0, T0)] + [np.abs(H0).max((1, 2))]
    amp += amp[1:3]
    der = np.einsum("p,npr,r->n", w, H0, w)
    for i, K in enumerate((T0, H1 * g, T1 * g, nd * H0, H1 * gm, T1 * gm)):
        for ab in range(4):
            ref = np.einsum("p,npr,r->n", W[ab // 2], K, W[ab % 2])
            if i == 3:
                ref = (der if ab in (0, 3) else -der) - kh ** 2 * ref
            assert np.max(np.abs(got[:, i, ab] - ref) / amp[i]) < 2.0 ** -24, (i, ab)
