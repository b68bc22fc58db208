"""The distance from which element pairs may be integrated on the FP32 pipe is the
caller's: pairs nearer than zfast are those of zfast = 0 (every pair in FP64) to the bit,
and wcs_info.zfast tells the distance in effect."""

import numpy as np
import pytest
import torch

from gpu_common import make_solver, to_np

pytestmark = pytest.mark.gpu

ELL = dict(family="ellipse", params={"ax": 1.0, "ay": 0.6}, N=700, k=None)


def columns(cols, **options):
    """Columns of the four stored operators, and the solver's info."""
    s = make_solver(ELL, precision=1, **options).assemble()
    eye = torch.zeros(s.N, len(cols), dtype=torch.complex128, device="cuda")
    eye[torch.as_tensor(cols), torch.arange(len(cols))] = 1.0
    out = [to_np(s.apply(op, eye)) for op in ("S", "D", "DT", "N")]
    info = s.info()
    x = s.geometry_sample(np.arange(s.N) * info["h"])
    s.close()
    return out, info, np.stack([x["x"], x["y"]], 1)


def test_pairs_below_the_callers_distance_stay_in_fp64():
    cols = [0, 100, 333, 699]
    ref, info, p = columns(cols, zfast=0.0)
    assert info["zfast"] == 0.0
    kh = info["k"] * info["h"]
    kR = info["k"] * np.hypot(*(p[:, None] - p[cols][None]).transpose(2, 0, 1))
    for z in (1.0e6, 60.0, 30.0):
        got, info, _ = columns(cols, zfast=z)
        assert info["zfast"] == pytest.approx(z + 2 * kh, rel=1e-12)
        near = kR < z                       # an entry's pairs have centres within k h of its nodes' distance
        assert near.all() == (z > kR.max())
        for g, r in zip(got, ref):
            assert np.array_equal(g[near], r[near])
            if not near.all():
                assert (g[~near] != r[~near]).any()


@pytest.mark.parametrize("kh,options,want", [(0.6, {}, 20.6), (0.6, dict(zfast=9.0), 20.6), (0.6, dict(zfast=500.0), 501.2),
                                             (1.5, {}, 1003.0), (1.5, dict(zfast=40.0), 43.0), (0.6, dict(precision=0), 0.0)])
def test_distance_in_effect(kh, options, want):
    s = make_solver(ELL, **dict(dict(precision=1), **options))
    s.mesh(ELL["N"], kh / s.info()["h"])
    assert s.info()["zfast"] == pytest.approx(want, rel=1e-12)
    s.close()


@pytest.mark.parametrize("ay,N,want", [(0.2, 300, "route"), (0.1, 420, "route"), (0.1, 380, "coarse"), (0.05, 400, "coarse")])
def test_elements_that_turn_by_a_radian(ay, N, want):
    """Curvature at the tip 1 / ay^2: the route starts at k R0 = 20 + k h while an element turns by
    less than a radian, and as on a coarse mesh beyond."""
    s = make_solver(dict(family="ellipse", params={"ax": 1.0, "ay": ay}, N=N, k=None), precision=1)
    i = s.info()
    s.close()
    kh = i["k"] * i["h"]
    assert (i["h"] / ay ** 2 <= 1.0) == (want == "route")
    assert i["zfast"] == pytest.approx(20 + kh if want == "route" else 1000 + 2 * kh, rel=1e-12)
