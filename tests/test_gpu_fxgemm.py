"""FP64 products on the tensor cores through fixed-point slices (fxgemm.cu),
through the public entry points that use them.

Each operand row is held to half a unit of its last digit, 2^-63 of its scale
2^E <= 2 rowmax, and digit pairs below 2^-62 of the scales are dropped, so with
a = max_k |A_ik|, b = max_k |B_kj| (componentwise magnitudes) the error of an
entry is at most 2k (2 * 2 * 2^-63 + 8 * 2^-62) 2a 2b <= k a b 2^-55, plus the
rounding of the result.  An FP64 dot product is only bounded by
2k 2^-53 sum |A||B|."""

import numpy as np
import pytest
import torch

import workloads
from gpu_common import built, make_solver, to_np

pytestmark = pytest.mark.gpu


def stored_operator(s, op):
    """The dense operator, exactly: products with unit vectors, few enough columns for the FP64 pipe."""
    N = s.N
    M = np.zeros((N, N), dtype=np.complex128)
    eye = torch.eye(N, dtype=torch.complex128, device="cuda")
    for j in range(0, N, 4):
        M[:, j:j + 4] = to_np(s.apply(op, eye[:, j:j + 4]))
    return M


# odd sizes around the tile (128 x 32 columns), the K = 32 stage and the K = 128 chunk
@pytest.mark.parametrize("N,B", [(320, 31), (320, 64), (385, 33), (513, 32), (640, 97)])
def test_operator_product_vs_extended_precision(N, B):
    built()
    w = dict(workloads.SMALL["superellipse_n320"], N=N)
    s = make_solver(w).assemble()
    rng = np.random.default_rng(N + B)
    X = rng.standard_normal((N, B)) + 1j * rng.standard_normal((N, B))
    X *= 10.0 ** rng.uniform(-6, 6, size=B)                     # column scales
    for op in ("S", "N"):
        A = stored_operator(s, op)
        ref = A.astype(np.clongdouble) @ X.astype(np.clongdouble)
        Y = to_np(s.apply(op, torch.tensor(X, device="cuda")))
        a = np.maximum(np.abs(A.real), np.abs(A.imag)).max(axis=1)[:, None]
        b = np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis=0)[None, :]
        bound = N * a * b * 2.0 ** -55 + 2.0 ** -51 * np.abs(ref).astype(float)
        assert np.all(np.abs(Y - ref).astype(float) <= bound)


@pytest.mark.parametrize("N,B", [(320, 48), (391, 40)])
def test_forward_and_adjoint_views(N, B):
    """C (K contiguous) and C^H (rows contiguous, conjugated) against the dense composition."""
    built()
    w = dict(workloads.SMALL["superellipse_n320"], N=N)
    s = make_solver(w).assemble()
    S, D, Dt, Nk = (stored_operator(s, op) for op in ("S", "D", "DT", "N"))
    h = s.info()["h"]
    G = np.zeros((N, N))
    i = np.arange(N)
    G[i, i], G[i, (i + 1) % N], G[(i + 1) % N, i] = 4 * h / 6, h / 6, h / 6
    C = (G / 2 + Dt) @ np.linalg.solve(G, G / 2 - D) + S @ np.linalg.solve(G, Nk)
    rng = np.random.default_rng(B)
    X = rng.standard_normal((N, B)) + 1j * rng.standard_normal((N, B))
    for op, M in (("C", C), ("CH", C.conj().T)):
        Y, ref = to_np(s.apply(op, torch.tensor(X, device="cuda"))), M @ X
        assert np.linalg.norm(Y - ref) <= 1e-12 * np.linalg.norm(ref)


def test_zero_and_non_finite_columns():
    """A zero column stays zero; a column that is not finite poisons itself and no other."""
    built()
    s = make_solver(dict(workloads.SMALL["superellipse_n320"])).assemble()
    N, B = s.N, 40
    X = np.random.default_rng(1).standard_normal((N, B)) + 0j
    clean = to_np(s.apply("S", torch.tensor(X, device="cuda")))
    X[:, 3] = 0.0
    X[7, 5], X[9, 6] = np.nan, np.inf
    Y = to_np(s.apply("S", torch.tensor(X, device="cuda")))
    assert np.all(Y[:, 3] == 0)
    assert not np.isfinite(Y[:, 5]).any() and not np.isfinite(Y[:, 6]).any()
    keep = [j for j in range(B) if j not in (3, 5, 6)]
    assert np.array_equal(Y[:, keep], clean[:, keep])
