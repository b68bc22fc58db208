"""Partial sums of split-K products that leave the FP32 range: an infinite partial gives an
infinite result, as an FP64 sum of the partials does, not NaN."""

import numpy as np
import pytest
import torch

from gpu_common import make_solver, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [600, 1111])
def test_overflowing_partial_is_infinite(N):
    # a large contour, so that the single layer's entries (~h^2) times a column of one huge
    # entry pass the FP32 range in the one split of K that holds it
    s = make_solver(dict(family="ellipse", params={"ax": 1.0e6, "ay": 7.0e5}, N=N, k=None), precision=1)
    s.assemble()
    j = N // 3
    x = torch.zeros(N, 1, dtype=torch.complex128, device="cuda")
    x[j] = 1.0
    a = to_np(s.apply("S", x))[:, 0]
    x[j] = big = 4.0 * 3.4e38 / np.max(np.abs(a))
    assert big < 3.0e38
    y = to_np(s.apply("S", x))[:, 0]
    s.close()
    over = 0
    for u, v in ((a.real, y.real), (a.imag, y.imag)):
        fits, exceeds = np.abs(u) * big < 3.0e38, np.abs(u) * big > 3.8e38   # second and third planes stay within the range
        assert np.all(np.abs(v[fits] - u[fits] * big) <= 1e-5 * 3.4e38)
        assert np.all(v[exceeds] == np.sign(u[exceeds]) * np.inf)
        over += exceeds.sum()
    assert over > 0
