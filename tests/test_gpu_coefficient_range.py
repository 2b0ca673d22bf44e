"""Coefficients far from 1 (whose squares leave FP64's range) scale the solution and
nothing else: a power of two in the stencil divides the iterates by it exactly, and
the residuals, which keep the right-hand side's size, stay as they are.

Tolerance 1e-12 of the larger of 1 and the value for histories, 1e-13 for
solutions: rounding may differ where a pass takes another route at that scale.
"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [-560, -530, 500, 600])
@pytest.mark.parametrize("dim,n,smoother,omega,c", [
    (2, 33, "rbgs", 1.0, (1.0, 1.0, 1.0)), (2, 129, "jacobi", 0.8, (1.0, 0.7, 1.0)),
    (2, 257, "rbgs", 1.0, (1.0, 1.0, 1.0)), (2, 513, "jacobi", 0.8, (0.7, 1.0, 1.0)),
    (3, 257, "rbgs", 1.0, (1.0, 1.0, 1.0))])
def test_node(dim, n, smoother, omega, c, shift):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    f = synth.uniform_rhs(dim, n, 98)
    got = []
    for e in (0, shift):
        s = Solver(dim, n, stencil=tuple(np.ldexp(c, e)), smoother=smoother, omega=omega, nu1=2, nu2=2, maxit=3)
        s.set_rhs(f)
        _, _, hist = s.solve(0.0, raise_on_noconv=False)
        got.append((hist, np.ldexp(s.get_solution(), e), s.residual_norm()))
    assert got[1][0].size == 4 and np.max(np.abs(got[1][0] - got[0][0]) / np.maximum(1.0, got[0][0])) <= 1e-12
    assert rel_err(got[1][1], got[0][1]) <= 1e-13
    assert abs(got[1][2] - got[0][2]) <= 1e-10 * got[0][2]


@pytest.mark.parametrize("shift", [-560, 520])
@pytest.mark.parametrize("n", [64, 256])
def test_cell(n, shift):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f = synth.uniform(99, (n, n))
    got = []
    for e in (0, shift):
        s = CCSolver(2, n, c=(np.ldexp(1.0, e),) * 2, sigma=np.ldexp(5.0, e), nu1=2, nu2=2, maxit=4)
        s.set_rhs(f)
        s.set_solution(None)
        _, _, hist = s.solve(0.0, raise_on_noconv=False)
        got.append((hist, np.ldexp(s.get_solution(), e)))
    assert got[1][0].size == 5 and np.max(np.abs(got[1][0] - got[0][0]) / np.maximum(1.0, got[0][0])) <= 1e-12
    assert rel_err(got[1][1], got[0][1]) <= 1e-13
