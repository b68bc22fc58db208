"""What a context keeps between calls must not cost a later call its memory: with a limit on
the context's buffers (wcs_memory_limit), a problem that runs in a new context runs in a
used one, tables that have no room are done without, and large buffers are given back."""

import numpy as np
import pytest
import torch

from gpu_common import colrel, to_np

pytestmark = pytest.mark.gpu

ELL = dict(ax=1.0, ay=0.6)


def new(precision, **options):
    from gpu_common import built
    built()
    from paper_2203_13283_gb300 import Solver
    return Solver(precision=precision, refine_tol=5e-7 if precision else 1e-10, **options).contour("ellipse", **ELL)


def setup(s, N, rank):
    s.mesh(N).assemble().skeleton(1e-6, max_rank=rank, seed=1, allow_cap=True)
    return s.factor()


def currents(s, N, B):
    return to_np(setup(s, N, N // 8).solve_planewaves(np.arange(B) * 0.05))


def smallest_limit(run, precision):
    """Bytes within 1% of the smallest limit under which run(new context) succeeds."""
    from paper_2203_13283_gb300 import WCSError

    def fits(limit):
        s = new(precision)
        s.memory(limit)
        try:
            run(s)
            return True
        except WCSError as e:
            assert e.status == 4
            return False
        finally:
            s.close()

    s = new(precision)
    run(s)
    hi = s.memory()
    s.close()
    lo = 0.1 * hi
    while not fits(hi):
        hi *= 1.02
    while hi - lo > 0.01 * hi:
        mid = 0.5 * (lo + hi)
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    return hi


@pytest.mark.parametrize("precision,N,used_N,used_B,used_rank", [(1, 1500, 700, 256, 600), (0, 900, 500, 256, 400)])
def test_a_used_context_has_the_room_of_a_new_one(precision, N, used_N, used_B, used_rank):
    limit = 1.1 * smallest_limit(lambda s: currents(s, N, 16), precision)
    s = new(precision)
    setup(s, used_N, used_rank).solve_planewaves(np.arange(used_B) * 0.01)
    s.farfield(torch.ones(used_N, 300, dtype=torch.complex128, device="cuda"), np.arange(300) * 0.02)
    s.solve_adjoint(torch.ones(used_N, 8, dtype=torch.complex128, device="cuda"), allow_unconverged=True)
    s.memory(limit)
    got = currents(s, N, 16)
    s.memory(0)
    s.close()
    t = new(precision)
    want = currents(t, N, 16)
    t.close()
    assert colrel(got, want) < (2e-6 if precision else 2e-10)


@pytest.mark.parametrize("precision,table,tol", [(1, 256 * 9 * 1500, 1e-7), (0, 16 * 16 * 33 * 33 * 7 * 47, 1e-12)])
def test_assembly_without_room_for_its_tables(precision, table, tol):
    def assemble(s):
        s.mesh(1500).assemble()

    s = new(precision)
    assemble(s)
    full = s.memory()
    x = torch.randn(1500, 4, dtype=torch.complex128, device="cuda", generator=torch.Generator(device="cuda").manual_seed(0))
    want = {op: to_np(s.apply(op, x)) for op in ("S", "D", "DT", "N", "CC")}
    s.close()
    limit = full - 0.9 * table
    s = new(precision)
    s.memory(limit)
    assemble(s)
    s.memory(0)
    for op, w in want.items():
        assert colrel(to_np(s.apply(op, x)), w) < tol, op
    s.close()


def test_large_buffers_are_given_back():
    s = new(1)
    currents(s, 16384, 256)
    before = s.memory()
    assert before > 25e9
    currents(s, 1000, 4)
    assert s.memory() < 2e9
    s.close()


def test_transform_plan_after_a_full_mesh():
    """The plan of a new length finds the room of the old mesh's operators."""
    s = new(0)
    s.mesh(1000).assemble()
    s.memory(s.memory() + (1 << 20))          # the operators of N = 1000 take 64 MB, the plan of N = 997 17 MB
    s.mesh(997)
    s.memory(0)
    x = torch.randn(997, 3, dtype=torch.complex128, device="cuda")
    s.assemble()
    f = np.fft.fft(to_np(x), axis=0) * to_np(s.circulant_eigs("CC"))[:, None]
    assert colrel(to_np(s.apply("CC", x)), np.fft.ifft(f, axis=0)) < 1e-12
    s.close()
