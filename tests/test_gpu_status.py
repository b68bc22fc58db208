"""An expired device wait reaches the caller: with the error flag of the bounded waits
raised (wcs_inject_timeout: nothing waits or fails on the device), every call whose
products may run on the tensor cores returns WCS_ERR_TIMEOUT, once; the calls after it
give the values of an untouched context."""

import numpy as np
import pytest
import torch

import workloads
from gpu_common import make_solver, to_np

pytestmark = pytest.mark.gpu

TIMEOUT = 8


@pytest.fixture(scope="module")
def solver():
    # FP64 form, sizes at which its products take the fixed-point route
    s = make_solver(workloads.SMALL["superellipse_n320"], refine_tol=1e-10)
    s.assemble()
    s.skeleton(1e-8, seed=1)
    s.factor()
    yield s
    s.close()


def block(n, B, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, B, dtype=torch.complex128, device="cuda", generator=g)


CALLS = {
    "apply_S": lambda s: s.apply("S", block(s.N, 40)),
    "apply_C": lambda s: s.apply("C", block(s.N, 40)),
    "apply_CH": lambda s: s.apply("CH", block(s.N, 40)),
    "apply_SKEL": lambda s: s.apply("SKEL", block(s.N, 128)),
    "woodbury": lambda s: s.woodbury_apply(block(s.N, 128)),
    "farfield": lambda s: s.farfield(block(s.N, 64), np.arange(180) * 0.03),
    "solve": lambda s: s.solve(block(s.N, 40)),
    "solve_adjoint": lambda s: s.solve_adjoint(block(s.N, 40)),
    "planewaves": lambda s: s.solve_planewaves(np.arange(40) * 0.1),
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_expired_wait_is_reported_once(solver, name):
    from paper_2203_13283_gb300._lib import WCSError, check
    call = CALLS[name]
    want = to_np(call(solver))
    check(solver.lib.wcs_inject_timeout(solver.h))
    with pytest.raises(WCSError) as ei:
        call(solver)
    assert ei.value.status == TIMEOUT
    assert np.array_equal(to_np(call(solver)), want)


def test_flag_raised_before_the_first_product():
    from paper_2203_13283_gb300._lib import WCSError, check
    s = make_solver(workloads.SMALL["superellipse_n320"])
    s.assemble()
    x = block(s.N, 40)
    want = to_np(s.apply("G", x))
    check(s.lib.wcs_inject_timeout(s.h))
    with pytest.raises(WCSError) as ei:
        s.apply("S", x)
    assert ei.value.status == TIMEOUT
    assert np.array_equal(to_np(s.apply("G", x)), want)
    s.close()
