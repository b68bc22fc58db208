"""The skeleton's basis over block widths and rows: U orthonormal to rounding, whatever the
split of its Gram products over CTAs (two CholeskyQR passes: their last Gram product's
roundings, a few hundred of 2^-53, bound |U^H U - I|: 1e-12).  FP64 form: the mixed form
shares these kernels, but projects block against block in split bf16."""

import numpy as np
import pytest
import torch

from gpu_common import make_solver, to_np

pytestmark = pytest.mark.gpu


# one pair; pairs of one CTA and one more (b = 10: 55, 11: 66); ragged row chunks and tiles
@pytest.mark.parametrize("N,block", [(97, 1), (255, 10), (256, 11), (257, 32), (700, 33), (1000, 64), (2100, 64)])
def test_skeleton_basis_is_orthonormal(N, block, tmp_path):
    s = make_solver(dict(family="ellipse", params={"ax": 1.0, "ay": 0.5}, N=N, k=None), block=block)
    s.assemble()
    rank = s.skeleton(1e-6, max_rank=min(N // 2, 130), seed=2, allow_cap=True)
    s.factor()
    path = str(tmp_path / "f.wcs")
    s.save(path)
    s.close()
    raw = np.fromfile(path, dtype=np.uint8)
    tail = 16 + 16 * rank * rank                     # trailer and capacitance inverse
    fac = raw[raw.size - tail - 3 * 16 * N * rank: raw.size - tail].view(np.complex128).reshape(3, rank, N)
    U = fac[0]
    assert np.max(np.abs(U.conj() @ U.T - np.eye(rank))) < 1e-12
